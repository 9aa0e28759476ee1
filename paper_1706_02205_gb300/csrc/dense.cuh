// Workspace of the dense product by split entries (dense.cu), sized once for
// all products of a refined solve.
#pragma once
#include "solver.cuh"

namespace kc {

struct DenseSplit {
    uint2* vf = nullptr;     // digits of the vectors
    double* coef = nullptr;  // scales, 16 per block of 128 columns
    double* part = nullptr;  // sums of every column range
    double* tab = nullptr;   // 2^(-j/256)
    int64_t per = 0;         // blocks per column range
    int splits = 0, nt = 0;
    // whether a product keeps FP64's accuracy row by row
    double* bmax = nullptr;           // largest value of every block, 16 per block
    double* scale = nullptr;             // per vector a power of two that takes |v| / sigma2 to float's range
    float *w = nullptr, *tw = nullptr;   // scale |v| and L L^T of it
    FactorEstimate LL;
    int* exact = nullptr;             // device: nonzero, this product is left to FP64
};
// P, val, diag: a factor L with L L^T like Theta (the preconditioner); norm2: the
// squared norms of the right-hand sides (device), near which the vectors are.
kc_status dense_split_init(DenseSplit& S, const kc_pattern* P, int prec, const void* val, const double* diag,
                           double sigma2, const double* norm2, int ns, Arena& A, cudaStream_t s);
// y = Theta v (point-major with stride ns <= 16, a power of two), closed-form Matern kernels (nu_code <= 2).
// Where *S.exact is nonzero afterwards y is not written: the caller forms it in FP64.
kc_status dense_theta_split(const DenseSplit& S, const double* x, int64_t N, int d, const KernelParams& kp,
                            const double* v, double* y, int ns, cudaStream_t s);

}  // namespace kc
