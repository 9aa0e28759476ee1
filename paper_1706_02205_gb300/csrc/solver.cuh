// Level-scheduled triangular-solve state shared by the solve and refinement.
#pragma once
#include "common.cuh"

namespace kc {

struct Solver {
    const kc_pattern* P = nullptr;
    int2* tasks = nullptr;
    const int64_t* ntasks_dev = nullptr;  // tasks of the backward solve
    int64_t ntasks = 0;                   // at most
    int rpt = 64;
    unsigned* cnt = nullptr;
    unsigned* gcnt = nullptr;
    double* acc = nullptr;
    unsigned long long* ticket = nullptr;
    int* status = nullptr;
    double* y = nullptr;
    float2* xf = nullptr;  // FP32 form: x as (hi, lo) pairs
    int nrhs_cap = 0;
    long long spin = 4000000000LL;
};

// out = L L^T in for point-major vectors of stride ns (a power of two <= 16) in
// positions order, in floats, with the workspace of one such product (tasks.cu).
struct FactorEstimate {
    const kc_pattern* P = nullptr;
    int prec = 0;
    const void* val = nullptr;
    const double* diag = nullptr;
    int ns = 1;
    int64_t* off = nullptr;
    int32_t* owner = nullptr;
    int64_t cap = 0;
    float *part = nullptr, *mid = nullptr;
    kc_status init(const kc_pattern* pat, int p, const void* v, const double* dg, int stride, Arena& A, cudaStream_t s);
    kc_status apply(const float* in, float* out, cudaStream_t s) const;
};

int64_t tasks_bound(const kc_pattern* P, int rpt);
kc_status build_tasks(const kc_pattern* P, int rpt, Arena& A, cudaStream_t s, int2** tasks_out,
                      const int64_t** count_out, int64_t* ntasks_out, bool adaptive = false);
kc_status solver_init(Solver& S, const kc_pattern* P, int nrhs_cap, const kc_opts* o, Arena& A, cudaStream_t s);
template <typename T>
kc_status solver_apply(Solver& S, const T* val, const double* diag, double diag_fallback, const double* rhs,
                       double* z, int nrhs, cudaStream_t s);
kc_status solver_check(Solver& S, cudaStream_t s);
// point-major copies with stride >= nrhs (0: nrhs); to_point_major zero-fills the padding
kc_status to_point_major(const double* b, const int32_t* perm, int64_t N, int nrhs, double* out, cudaStream_t s,
                         int stride = 0);
kc_status from_point_major(const double* xp, const int32_t* perm, int64_t N, int nrhs, double* x, cudaStream_t s,
                           int stride = 0);

}  // namespace kc
