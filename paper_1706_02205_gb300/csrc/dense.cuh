// Workspace of the dense product by split entries (dense.cu), sized once for
// all products of a refined solve.
#pragma once
#include "common.cuh"

namespace kc {

struct DenseSplit {
    uint2* vf = nullptr;     // digits of the vectors
    double* coef = nullptr;  // scales, 16 per block of 128 columns
    double* part = nullptr;  // sums of every column range
    double* tab = nullptr;   // 2^(-j/256)
    int64_t per = 0;         // blocks per column range
    int splits = 0, nt = 0;
};
kc_status dense_split_init(DenseSplit& S, int64_t N, int ns, Arena& A, cudaStream_t s);
// y = Theta v (point-major with stride ns <= 16, a power of two), closed-form Matern kernels (nu_code <= 2)
kc_status dense_theta_split(const DenseSplit& S, const double* x, int64_t N, int d, const KernelParams& kp,
                            const double* v, double* y, int ns, cudaStream_t s);

}  // namespace kc
