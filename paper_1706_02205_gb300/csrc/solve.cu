// a7: L L^T x = b with the sparse factor (task (2) of Section 1), as two
// sync-free level-scheduled triangular solves in one persistent launch each.
//
// Forward  L y = b:   y_j = (b_j - sum_{k in R_j} L_jk y_k) / L_jj, one warp per
//                     row, rows in (level, index) order; row j waits for the
//                     values of its R_j.
// Backward L^T x = y: x_i = (y_i - sum_{j in C_i} L_ji x_j) / L_ii, over the
//                     CSC columns in reverse level order; wide columns are cut
//                     into chunks of rows, each chunk stores its partial sums
//                     in a slot of its own; the last chunk to finish of every
//                     group of 32 adds its group's slots, and the last group
//                     of a column to finish adds the group sums and finishes
//                     x_i.  Every sum runs in a fixed order across the lanes
//                     of a warp, so every result repeats bit for bit.
//
// Vectors are point-major inside with a power-of-two stride NR >= nrhs
// (v[k * NR + r]), so one point's right-hand sides are one aligned run that a
// lane gathers with 16-byte loads.  A lane owns entries of the row (or rows of
// the column): their columns and values are loaded first, then their points'
// values in a few rounds; a value not yet set is polled (await_words), which
// for the early, coarse points of a row never happens, so their products are
// done while the last ones are still on their way.  The warp reduces its NR
// partial sums with a reduce-scatter.  A dropped pivot (L_ii = 0) uses
// sqrt(Theta_ii).
//
// Bound by the chain of dependency levels (each a store, a poll, the warp's
// reduction and a division) and, at 16 right-hand sides, by the gathers (128
// bytes an entry from L1 and L2).  Values that carry their own readiness,
// against ready flags with fences on both sides: 2000 points, one right-hand
// side 1.0 -> 0.5 ms; 100,003 points 3.9 -> 1.4; 2^20 points, rho = 3, 11.0 ->
// 6.8 (one) and 14.3 -> 12.0 (16, FP32 form), 22.6 -> 18.4 (16, FP64).
//
// Arithmetic.  FP64 form: vectors, products and sums in FP64.  FP32 form (L in
// FP32): the GB300's FP64 pipe is a small fraction of its FP32 rate, so the
// vectors are kept as pairs of floats (hi, lo) with hi + lo the FP64 value to
// about 2^-48, every product L_jk (hi + lo) is formed with TwoProduct (fmaf)
// plus the small L_jk lo term, and the sums are compensated (TwoSum, the
// scheme of Ogita, Rump and Oishi's Dot2); each row's result is formed in
// FP64 and split back into a pair.  The solution is about 2^-45 accurate
// relative to the sums' magnitudes, where FP64 gives 2^-53.
#include <type_traits>

#include "pairs.cuh"
#include "solver.cuh"

namespace kc {

// Right-hand sides a lane of the FP32-form kernels keeps (an entry's NR are
// split over NR / KC_SOLVE_NRL lanes), and the resident 256-thread CTAs per
// SM their register budget is cut for.
#ifndef KC_SOLVE_NRL
#define KC_SOLVE_NRL 8
#endif
#ifndef KC_SOLVE_MINB
#define KC_SOLVE_MINB 3
#endif

// Right-hand sides up to which a row's b, y and pivot are fetched before its
// waits (beyond, the registers they hold cost more).
#ifndef KC_SOLVE_EARLY
#define KC_SOLVE_EARLY 4
#endif

// Warps per row of a dependency level that a solve launches at most.
#ifndef KC_SOLVE_WAVES
#define KC_SOLVE_WAVES 8.0
#endif

// Longest back-off (ns) between two polls of a value.
template <int NR>
constexpr int BACKOFF_MAX = NR > 4 ? 128 : 64;

template <typename T>
struct SolveArgs {
    int64_t N;
    const int64_t* __restrict__ rowptr;
    const int32_t* __restrict__ col;
    const int64_t* __restrict__ colptr;
    const int32_t* __restrict__ rowidx;
    const int64_t* __restrict__ slot;
    const int32_t* __restrict__ order;
    const int2* __restrict__ tasks;
    const int64_t* __restrict__ ntasks;  // device
    int rpt;
    const T* __restrict__ val;
    const double* __restrict__ diag;
    double diag_fallback;
    const double* b;  // point-major input
    double* y;        // point-major output of the forward solve / input of backward (FP64 form)
    double* x;        // point-major output of the backward solve
    float2* yf;       // FP32 form: y as (hi, lo) pairs
    float2* xf;       // FP32 form: x as (hi, lo) pairs (gathered by later columns; x above gets FP64)
    double* acc;      // partial sums of the chunks of wide columns: NR per task, at the task's index
    unsigned* cnt;    // finished chunk groups per column (backward)
    unsigned* gcnt;   // finished chunks per group of 32, at the group's first task
    unsigned long long* ticket;
    int* status;
    long long spin_limit;
};

// A point's vector values carry their own readiness: the buffers start as all
// ones (a NaN no value takes, see word_of), every value is stored once as one
// 8-byte word, and whoever needs it loads it until it is set.  A row's result
// then reaches the rows that wait for it in one store and one load; with ready
// flags it took a fence before the flag, the poll, another fence and only then
// the gathers (2^20 points, rho = 3, one right-hand side, FP32 form: 10.6 ms).


// 16 (8) bytes of vector values through L1: coarse points are gathered by nearly
// every row.  A line cached before its values were set only sends the reader to
// the polling loads below, which go to L2.
__device__ __forceinline__ ulonglong2 ld_first(const ulonglong2* p) {
    ulonglong2 v;
    asm volatile("ld.global.ca.v2.u64 {%0, %1}, [%2];" : "=l"(v.x), "=l"(v.y) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ unsigned long long ld_first(const unsigned long long* p) {
    unsigned long long v;
    asm volatile("ld.global.ca.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ unsigned long long ld_again(const unsigned long long* p) {
    unsigned long long v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void st_value(unsigned long long* p, unsigned long long v) {
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
// The word of a value; a NaN that happens to be all ones in its first half
// becomes the usual one, so that no value looks unset.
__device__ __forceinline__ unsigned long long word_of(double v) {
    const unsigned long long w = (unsigned long long)__double_as_longlong(v);
    return (unsigned)(w >> 32) == 0xffffffffu ? 0x7fffffffffffffffull : w;
}
__device__ __forceinline__ unsigned long long word_of(float2 v) {
    const unsigned hi = __float_as_uint(v.x);
    return ((unsigned long long)__float_as_uint(v.y) << 32) | (hi == 0xffffffffu ? 0x7fffffffu : hi);
}
// FP64: the high half tells; pairs: hi, in the low half
template <typename V>
__device__ __forceinline__ bool is_unset(unsigned long long w);
template <>
__device__ __forceinline__ bool is_unset<double>(unsigned long long w) { return (unsigned)(w >> 32) == 0xffffffffu; }
template <>
__device__ __forceinline__ bool is_unset<float2>(unsigned long long w) { return (unsigned)w == 0xffffffffu; }

// N words of a point's values, loaded once (no wait)
template <int N>
__device__ __forceinline__ void ld_words(const unsigned long long* p, unsigned long long (&w)[N]) {
    if constexpr (N == 1) {
        w[0] = ld_first(p);
    } else {
#pragma unroll
        for (int q = 0; q < N / 2; ++q) {
            const ulonglong2 x = ld_first((const ulonglong2*)p + q);
            w[2 * q] = x.x;
            w[2 * q + 1] = x.y;
        }
    }
}
// Bounded wait (backoff) until all of them are set; false when the budget ran
// out or the kernel is stopping.
template <typename V, int NR, int N>
__device__ __forceinline__ bool await_words(const unsigned long long* p, unsigned long long (&w)[N], const int* status,
                                            long long limit) {
    bool open = false;
#pragma unroll
    for (int q = 0; q < N; ++q) open |= is_unset<V>(w[q]);
    if (!open) return true;
    const long long t0 = clock64();
    unsigned ns = 32;
    for (int poll = 1;; ++poll) {
        w[0] = ld_again(p);  // one word stands for the point until it is set
        if (!is_unset<V>(w[0])) {
            open = false;
#pragma unroll
            for (int q = 1; q < N; ++q) {
                w[q] = ld_again(p + q);
                open |= is_unset<V>(w[q]);
            }
            if (!open) return true;
        }
        if (clock64() - t0 > limit || ((poll & 15) == 0 && ld_volatile_s32(status) != 0)) return false;
        __nanosleep(ns);  // back off so waiting warps do not flood L2 with polls
        if (ns < BACKOFF_MAX<NR>) ns <<= 1;
    }
}

// Warp reduce-scatter of NR partial sums per lane: each level halves the
// values a lane keeps (offsets 16, 8, ...), plain sums finish the rest.  The
// lane ends with the full sum of right-hand side rhs_of_lane<NR>(lane).
template <int NR>
__device__ __forceinline__ double reduce_scatter(double (&v)[NR], int lane) {
    const unsigned FULL = 0xffffffffu;
#pragma unroll
    for (int h = NR / 2, o = 16; h >= 1; h >>= 1, o >>= 1) {
        const bool up = (lane & o) != 0;
#pragma unroll
        for (int q = 0; q < h; ++q) {
            const double send = up ? v[q] : v[q + h];
            const double keep = up ? v[q + h] : v[q];
            v[q] = keep + __shfl_xor_sync(FULL, send, o);
        }
    }
    constexpr int L = NR == 1 ? 0 : NR == 2 ? 1 : NR == 4 ? 2 : NR == 8 ? 3 : 4;
#pragma unroll
    for (int o = 16 >> L; o >= 1; o >>= 1) v[0] += __shfl_xor_sync(FULL, v[0], o);
    return v[0];
}
template <int NR>
__device__ __forceinline__ int rhs_of_lane(int lane) {
    int r = 0;
#pragma unroll
    for (int h = NR / 2, o = 16; h >= 1; h >>= 1, o >>= 1)
        if (lane & o) r += h;
    return r;
}
// one writer per right-hand side: the lanes sharing r differ in the low bits
template <int NR>
__device__ __forceinline__ bool rhs_writer(int lane) {
    return (lane & (32 / NR - 1)) == 0;
}

// Entries in flight per lane while gathering: at most 32 doubles.
template <int NR>
struct Depth {
    static constexpr int E = NR >= 4 ? 32 / NR : 8;
};

// acc[r] += w[u] * v[k[u] * NR + r] for the D entries in order, E gathers at a
// time, each point waited for where it is not solved yet.  False: a wait ran out.
template <int NR, int D>
__device__ __forceinline__ bool gather_fma(const double* v, const int (&k)[D], const double (&w)[D], double (&acc)[NR],
                                           const int* status, long long limit) {
    constexpr int E = Depth<NR>::E < D ? Depth<NR>::E : D;
    bool ok = true;
#pragma unroll
    for (int u0 = 0; u0 < D; u0 += E) {
        unsigned long long g[E][NR];
#pragma unroll
        for (int q = 0; q < E; ++q)
            if (k[u0 + q] >= 0) ld_words<NR>((const unsigned long long*)v + (int64_t)k[u0 + q] * NR, g[q]);
#pragma unroll
        for (int q = 0; q < E; ++q)
            if (k[u0 + q] >= 0) {  // the FP64 pipe is scarce: no products for empty slots
                if (ok)
                    ok = await_words<double, NR, NR>((const unsigned long long*)v + (int64_t)k[u0 + q] * NR, g[q], status,
                                                 limit);
#pragma unroll
                for (int r = 0; r < NR; ++r)
                    acc[r] = fma(w[u0 + q], __longlong_as_double((long long)g[q][r]), acc[r]);
            }
    }
    return ok;
}

// Sum over cnt slots of NR doubles (slot p0, p0 + stride, ...) in a fixed
// order: lane l takes right-hand side l % NR and every (32 / NR)-th slot from
// l / NR on; the lanes of one right-hand side then add their sums by a fixed
// butterfly.  Every lane returns the total of right-hand side lane % NR.
template <int NR>
__device__ __forceinline__ double combine_slots(const double* part, int64_t p0, int64_t stride, int cnt, int lane) {
    constexpr int LP = 32 / NR;
    const int r = lane % NR;
    double s = 0.0;
    for (int k = lane / NR; k < cnt; k += LP) s += __ldcg(&part[(p0 + (int64_t)k * stride) * NR + r]);
#pragma unroll
    for (int o = 16; o >= NR; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    return s;
}

// A chunk c of column i (task index ti, nch > 1 chunks) with its partial sums
// already in its slot: counts it in its group of 32 chunks; the group's last
// chunk adds the group's slots and leaves the sum in the group's first slot;
// the column's last group adds the group sums.  Returns true (and the total
// of right-hand side lane % NR in `total`) when this warp finishes column i.
template <int NR>
__device__ __forceinline__ bool combine_chunks(double* part, unsigned* gcnt, unsigned* cnt, int i, int64_t ti, int c,
                                               unsigned nch, int lane, double& total) {
    const unsigned FULL = 0xffffffffu;
    const int64_t base = ti - c;
    const int g = c >> 5, ng = (int)((nch + 31) >> 5);
    const int gsz = (int)min(32u, nch - 32u * (unsigned)g);
    unsigned prev = 0;
    fence_acq_rel_gpu();
    __syncwarp();
    if (lane == 0) prev = atomicAdd(&gcnt[base + 32 * g], 1u);
    prev = __shfl_sync(FULL, prev, 0);
    if ((int)prev != gsz - 1) return false;
    fence_acq_rel_gpu();  // acquire: the group's slots are visible
    double gs = combine_slots<NR>(part, base + 32 * g, 1, gsz, lane);
    if (ng == 1) {
        total = gs;
        return true;
    }
    if (lane < NR) part[(base + 32 * g) * NR + lane] = gs;
    fence_acq_rel_gpu();
    __syncwarp();
    if (lane == 0) prev = atomicAdd(&cnt[i], 1u);
    prev = __shfl_sync(FULL, prev, 0);
    if ((int)prev != ng - 1) return false;
    fence_acq_rel_gpu();
    total = combine_slots<NR>(part, base, 32, ng, lane);
    return true;
}

template <typename T, int NR>
__global__ void __launch_bounds__(256, 2) fwd_solve_k(SolveArgs<T> A) {
    constexpr int D = 8;  // entries of R_j per lane per round
    const int lane = lane_id();
    const unsigned FULL = 0xffffffffu;
    for (;;) {
        unsigned long long t = 0;
        if (lane == 0) t = atomicAdd(A.ticket, 1ULL);
        t = __shfl_sync(FULL, t, 0);
        if ((int64_t)t >= A.N) return;
        if (ld_volatile_s32(A.status) != 0) return;
        const int j = A.order[t];
        const int64_t a = A.rowptr[j];
        const int n = (int)(A.rowptr[j + 1] - 1 - a);
        // what finishes the row, fetched before the waits
        const int r = rhs_of_lane<NR>(lane);
        const bool wr = rhs_writer<NR>(lane);
        double bj = 0.0, dj = 0.0;
        if constexpr (NR <= KC_SOLVE_EARLY) {
            if (wr) bj = A.b[(int64_t)j * NR + r];
            dj = A.diag[j];
        }
        double acc[NR];
#pragma unroll
        for (int r = 0; r < NR; ++r) acc[r] = 0.0;
        for (int e0 = 0; e0 < n; e0 += 32 * D) {
            int kk[D];
#pragma unroll
            for (int u = 0; u < D; ++u) {
                const int e = e0 + lane + 32 * u;
                kk[u] = e < n ? __ldg(&A.col[a + e]) : -1;
            }
            double w[D];  // static data: loaded before the wait
#pragma unroll
            for (int u = 0; u < D; ++u) w[u] = kk[u] >= 0 ? (double)__ldg(&A.val[a + e0 + lane + 32 * u]) : 0.0;
            if (!__all_sync(FULL, gather_fma<NR, D>(A.y, kk, w, acc, A.status, A.spin_limit))) {
                if (lane == 0) atomicCAS(A.status, 0, DEV_TIMEOUT);
                return;
            }
        }
        const double s = reduce_scatter<NR>(acc, lane);
        if (wr) {
            if constexpr (NR > KC_SOLVE_EARLY) {
                bj = A.b[(int64_t)j * NR + r];
                dj = A.diag[j];
            }
            if (!(dj > 0.0)) dj = A.diag_fallback;
            st_value((unsigned long long*)A.y + (int64_t)j * NR + r, word_of((bj - s) / dj));
        }
    }
}

template <typename T, int NR>
__global__ void __launch_bounds__(256, 2) bwd_solve_k(SolveArgs<T> A) {
    constexpr int D = 4;  // rows of the chunk per lane per round
    const int lane = lane_id();
    const unsigned FULL = 0xffffffffu;
    for (;;) {
        unsigned long long t = 0;
        if (lane == 0) t = atomicAdd(A.ticket, 1ULL);
        t = __shfl_sync(FULL, t, 0);
        const int64_t nt = __ldg(A.ntasks);
        if ((int64_t)t >= nt) return;
        if (ld_volatile_s32(A.status) != 0) return;
        const int64_t ti = nt - 1 - (int64_t)t;
        const int2 tk = A.tasks[ti];
        const int i = tk.x, c = tk.y;
        const int64_t c0 = A.colptr[i], c1 = A.colptr[i + 1];
        const int64_t m = c1 - c0 - 1;
        const unsigned nch = m <= 0 ? 1u : (unsigned)((m + A.rpt - 1) / A.rpt);
        const int64_t qs = c0 + 1 + (int64_t)c * A.rpt;
        const int nq = (int)(min(c1, qs + A.rpt) - qs);
        // what finishes a column of one chunk, fetched before the waits
        int r = rhs_of_lane<NR>(lane);
        bool wr = rhs_writer<NR>(lane);
        double yi = 0.0, di = 0.0;
        if constexpr (NR <= KC_SOLVE_EARLY) {
            if (wr) yi = A.y[(int64_t)i * NR + r];
            di = A.diag[i];
        }
        double acc[NR];
#pragma unroll
        for (int r = 0; r < NR; ++r) acc[r] = 0.0;
        for (int q0 = 0; q0 < nq; q0 += 32 * D) {
            int jj[D];
            int64_t pp[D];
#pragma unroll
            for (int u = 0; u < D; ++u) {
                const int q = q0 + lane + 32 * u;
                jj[u] = q < nq ? __ldg(&A.rowidx[qs + q]) : -1;
                pp[u] = q < nq ? __ldg(&A.slot[qs + q]) : 0;
            }
            double w[D];  // static data: loaded before the wait
#pragma unroll
            for (int u = 0; u < D; ++u) w[u] = jj[u] >= 0 ? (double)__ldg(&A.val[pp[u]]) : 0.0;
            if (!__all_sync(FULL, gather_fma<NR, D>(A.x, jj, w, acc, A.status, A.spin_limit))) {
                if (lane == 0) atomicCAS(A.status, 0, DEV_TIMEOUT);
                return;
            }
        }
        double s = reduce_scatter<NR>(acc, lane);
        bool finish = true;
        if (nch > 1) {
            if (wr) A.acc[ti * NR + r] = s;
            finish = combine_chunks<NR>(A.acc, A.gcnt, A.cnt, i, ti, c, nch, lane, s);
            wr = lane < NR;  // the combined sums: right-hand side lane % NR
            r = lane % NR;
            if constexpr (NR <= KC_SOLVE_EARLY) yi = A.y[(int64_t)i * NR + r];
        }
        if (finish && wr) {
            if constexpr (NR > KC_SOLVE_EARLY) {
                yi = A.y[(int64_t)i * NR + r];
                di = A.diag[i];
            }
            if (!(di > 0.0)) di = A.diag_fallback;
            st_value((unsigned long long*)A.x + (int64_t)i * NR + r, word_of((yi - s) / di));
        }
    }
}

// ------------------------------------------------ FP32 form: float pairs
// Lane layout of the pair kernels: an entry's NR right-hand sides are split
// over P lanes of NRL each (NR = 16: two lanes of 8; else one lane), so a lane
// keeps NRL compensated sums and gathers NRL pairs per entry: half the
// registers of one lane per entry at NR = 16, hence twice the resident warps.
template <int NR>
struct PairLayout {
    static constexpr int NRL = NR > KC_SOLVE_NRL ? KC_SOLVE_NRL : NR;  // right-hand sides per lane
    static constexpr int P = NR / NRL;           // lanes per entry (1 or 2)
    static constexpr int SLOTS = 32 / P;         // entries per warp and round
    static constexpr int L = NRL == 1 ? 0 : NRL == 2 ? 1 : NRL == 4 ? 2 : 3;  // halving levels
};

// Reduce-scatter of the NRL (s, c) pairs over the lanes holding the same block
// of right-hand sides (offsets 16, 8, ... down to P); returns the FP64 sum of
// right-hand side pair_rhs<NR>(lane).
template <int NR>
__device__ __forceinline__ double reduce_scatter_pair(float (&s)[PairLayout<NR>::NRL],
                                                      float (&c)[PairLayout<NR>::NRL], int lane) {
    using PL = PairLayout<NR>;
    const unsigned FULL = 0xffffffffu;
#pragma unroll
    for (int h = PL::NRL / 2, o = 16; h >= 1; h >>= 1, o >>= 1) {
        const bool up = (lane & o) != 0;
#pragma unroll
        for (int q = 0; q < h; ++q) {
            const float ss = up ? s[q] : s[q + h], sc = up ? c[q] : c[q + h];
            const float ks = up ? s[q + h] : s[q], kc = up ? c[q + h] : c[q];
            const float rs = __shfl_xor_sync(FULL, ss, o), rc = __shfl_xor_sync(FULL, sc, o);
            s[q] = ks;
            c[q] = kc;
            pair_merge(s[q], c[q], rs, rc);
        }
    }
#pragma unroll
    for (int o = 16 >> PL::L; o >= PL::P; o >>= 1) {
        const float rs = __shfl_xor_sync(FULL, s[0], o), rc = __shfl_xor_sync(FULL, c[0], o);
        pair_merge(s[0], c[0], rs, rc);
    }
    return (double)s[0] + (double)c[0];
}
template <int NR>
__device__ __forceinline__ int pair_rhs(int lane) {
    using PL = PairLayout<NR>;
    int r = (lane & (PL::P - 1)) * PL::NRL;
#pragma unroll
    for (int h = PL::NRL / 2, o = 16; h >= 1; h >>= 1, o >>= 1)
        if (lane & o) r += h;
    return r;
}
// one writer per right-hand side: the lanes sharing one differ only in the
// bits between the block bits and the halving bits
template <int NR>
__device__ __forceinline__ bool pair_writer(int lane) {
    using PL = PairLayout<NR>;
    return (lane & ((32 >> PL::L) - 1) & ~(PL::P - 1)) == 0;
}

// (s, c)[r] += w[u] * v[k[u]][block + r] for the D entries in order, E gathers
// at a time, nothing for empty slots; each point waited for where it is not
// solved yet.  False: a wait ran out.
template <int NR, int D>
__device__ __forceinline__ bool gather_pair_add(const float2* v, const int (&k)[D], const float (&w)[D], int block,
                                                float (&s)[PairLayout<NR>::NRL], float (&c)[PairLayout<NR>::NRL],
                                                const int* status, long long limit) {
    constexpr int NRL = PairLayout<NR>::NRL;
    constexpr int E0 = NRL >= 2 ? 16 / NRL : 8;  // at most 16 pairs in flight per lane
    constexpr int E = E0 < D ? E0 : D;
    bool ok = true;
#pragma unroll
    for (int u0 = 0; u0 < D; u0 += E) {
        unsigned long long g[E][NRL];
#pragma unroll
        for (int q = 0; q < E; ++q)
            if (k[u0 + q] >= 0)
                ld_words<NRL>((const unsigned long long*)v + (int64_t)k[u0 + q] * NR + block, g[q]);
#pragma unroll
        for (int q = 0; q < E; ++q)
            if (k[u0 + q] >= 0) {
                if (ok)
                    ok = await_words<float2, NR, NRL>((const unsigned long long*)v + (int64_t)k[u0 + q] * NR + block, g[q],
                                                  status, limit);
#pragma unroll
                for (int r = 0; r < NRL; ++r)
                    pair_add(s[r], c[r], w[u0 + q], __uint_as_float((unsigned)g[q][r]),
                             __uint_as_float((unsigned)(g[q][r] >> 32)));
            }
    }
    return ok;
}

template <int NR>
__global__ void __launch_bounds__(256, KC_SOLVE_MINB) fwd_solve_pair_k(SolveArgs<float> A) {
    using PL = PairLayout<NR>;
    constexpr int D = PL::NRL >= 8 ? 6 : 8;  // entries per lane and round (within 80 registers)
    const int lane = lane_id();
    const int el = lane / PL::P, block = (lane & (PL::P - 1)) * PL::NRL;
    const unsigned FULL = 0xffffffffu;
    for (;;) {
        unsigned long long t = 0;
        if (lane == 0) t = atomicAdd(A.ticket, 1ULL);
        t = __shfl_sync(FULL, t, 0);
        if ((int64_t)t >= A.N) return;
        if (ld_volatile_s32(A.status) != 0) return;
        const int j = A.order[t];
        const int64_t a = A.rowptr[j];
        const int n = (int)(A.rowptr[j + 1] - 1 - a);
        // what finishes the row, fetched before the waits
        const int r = pair_rhs<NR>(lane);
        const bool wr = pair_writer<NR>(lane);
        double bj = 0.0, dj = 0.0;
        if constexpr (NR <= KC_SOLVE_EARLY) {
            if (wr) bj = A.b[(int64_t)j * NR + r];
            dj = A.diag[j];
        }
        float s[PL::NRL], c[PL::NRL];
#pragma unroll
        for (int r = 0; r < PL::NRL; ++r) s[r] = c[r] = 0.f;
        for (int e0 = 0; e0 < n; e0 += PL::SLOTS * D) {
            int kk[D];
            float w[D];  // static data: loaded before the wait
#pragma unroll
            for (int u = 0; u < D; ++u) {
                const int e = e0 + el + PL::SLOTS * u;
                kk[u] = e < n ? __ldg(&A.col[a + e]) : -1;
                w[u] = e < n ? __ldg(&A.val[a + e]) : 0.f;
            }
            if (!__all_sync(FULL, gather_pair_add<NR, D>(A.yf, kk, w, block, s, c, A.status, A.spin_limit))) {
                if (lane == 0) atomicCAS(A.status, 0, DEV_TIMEOUT);
                return;
            }
        }
        const double sum = reduce_scatter_pair<NR>(s, c, lane);
        if (wr) {
            if constexpr (NR > KC_SOLVE_EARLY) {
                bj = A.b[(int64_t)j * NR + r];
                dj = A.diag[j];
            }
            if (!(dj > 0.0)) dj = A.diag_fallback;
            st_value((unsigned long long*)A.yf + (int64_t)j * NR + r, word_of(pair_of((bj - sum) / dj)));
        }
    }
}

template <int NR>
__global__ void __launch_bounds__(256, KC_SOLVE_MINB) bwd_solve_pair_k(SolveArgs<float> A) {
    using PL = PairLayout<NR>;
    constexpr int D = 4;
    const int lane = lane_id();
    const int el = lane / PL::P, block = (lane & (PL::P - 1)) * PL::NRL;
    const unsigned FULL = 0xffffffffu;
    for (;;) {
        unsigned long long t = 0;
        if (lane == 0) t = atomicAdd(A.ticket, 1ULL);
        t = __shfl_sync(FULL, t, 0);
        const int64_t nt = __ldg(A.ntasks);
        if ((int64_t)t >= nt) return;
        if (ld_volatile_s32(A.status) != 0) return;
        const int64_t ti = nt - 1 - (int64_t)t;
        const int2 tk = A.tasks[ti];
        const int i = tk.x, ch = tk.y;
        const int64_t c0 = A.colptr[i], c1 = A.colptr[i + 1];
        const int64_t m = c1 - c0 - 1;
        const unsigned nch = m <= 0 ? 1u : (unsigned)((m + A.rpt - 1) / A.rpt);
        const int64_t qs = c0 + 1 + (int64_t)ch * A.rpt;
        const int nq = (int)(min(c1, qs + A.rpt) - qs);
        // what finishes a column of one chunk, fetched before the waits
        int r = pair_rhs<NR>(lane);
        bool wr = pair_writer<NR>(lane);
        float2 yi = make_float2(0.f, 0.f);
        double di = 0.0;
        if constexpr (NR <= KC_SOLVE_EARLY) {
            if (wr) yi = A.yf[(int64_t)i * NR + r];
            di = A.diag[i];
        }
        float s[PL::NRL], c[PL::NRL];
#pragma unroll
        for (int r = 0; r < PL::NRL; ++r) s[r] = c[r] = 0.f;
        for (int q0 = 0; q0 < nq; q0 += PL::SLOTS * D) {
            int jj[D];
            float w[D];  // static data: loaded before the wait
#pragma unroll
            for (int u = 0; u < D; ++u) {
                const int q = q0 + el + PL::SLOTS * u;
                jj[u] = q < nq ? __ldg(&A.rowidx[qs + q]) : -1;
                w[u] = q < nq ? __ldg(&A.val[__ldg(&A.slot[qs + q])]) : 0.f;
            }
            if (!__all_sync(FULL, gather_pair_add<NR, D>(A.xf, jj, w, block, s, c, A.status, A.spin_limit))) {
                if (lane == 0) atomicCAS(A.status, 0, DEV_TIMEOUT);
                return;
            }
        }
        double sum = reduce_scatter_pair<NR>(s, c, lane);
        bool finish = true;
        if (nch > 1) {
            if (wr) A.acc[ti * NR + r] = sum;
            finish = combine_chunks<NR>(A.acc, A.gcnt, A.cnt, i, ti, ch, nch, lane, sum);
            wr = lane < NR;  // the combined sums: right-hand side lane % NR
            r = lane % NR;
            if constexpr (NR <= KC_SOLVE_EARLY) yi = A.yf[(int64_t)i * NR + r];
        }
        if (finish && wr) {
            if constexpr (NR > KC_SOLVE_EARLY) {
                yi = A.yf[(int64_t)i * NR + r];
                di = A.diag[i];
            }
            if (!(di > 0.0)) di = A.diag_fallback;
            const double xi = (value_of(yi) - sum) / di;
            st_value((unsigned long long*)A.xf + (int64_t)i * NR + r, word_of(pair_of(xi)));
            A.x[(int64_t)i * NR + r] = xi;
        }
    }
}

// out[k * stride + r] = b[r * N + perm[k]] for r < nrhs, 0 for nrhs <= r < stride
__global__ void to_point_major_k(const double* __restrict__ b, const int32_t* __restrict__ perm, int64_t N, int nrhs,
                                 int stride, double* __restrict__ out) {
    int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t < N * stride) {
        int64_t k = t / stride;
        int r = (int)(t % stride);
        out[t] = r < nrhs ? b[(int64_t)r * N + perm[k]] : 0.0;
    }
}
__global__ void from_point_major_k(const double* __restrict__ xp, const int32_t* __restrict__ perm, int64_t N,
                                   int nrhs, int stride, double* __restrict__ x) {
    int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t < N * nrhs) {
        int64_t k = t / nrhs;
        int r = (int)(t % nrhs);
        x[(int64_t)r * N + perm[k]] = xp[k * stride + r];
    }
}

// Rows of a column per backward-solve task (wider columns are cut into chunks
// whose sums the column's last chunk adds in chunk order).
#ifndef KC_SOLVE_ROWS
#define KC_SOLVE_ROWS 128
#endif

kc_status solver_init(Solver& S, const kc_pattern* P, int nrhs_cap, const kc_opts* o, Arena& A, cudaStream_t s) {
    S.P = P;
    S.rpt = (o && o->rows_per_task > 0) ? o->rows_per_task : 0;
    if (S.rpt == 0) {
        // Few right-hand sides and more chunks per level than resident warps: longer
        // chunks, so that a column has fewer sums to combine (2^20 points, rho = 3,
        // one right-hand side: 128 rows 7.9 ms, 256 6.7, 512 6.7; 16 right-hand
        // sides: 12.1, 12.4, 13.9).
        S.rpt = KC_SOLVE_ROWS;
        const int64_t warps = (int64_t)sm_count() * 32;
        if (nrhs_cap <= 4 && tasks_bound(P, KC_SOLVE_ROWS) > warps * (P->depth > 0 ? P->depth : 1)) S.rpt = 2 * KC_SOLVE_ROWS;
    }
    if (o && o->spin_limit_cycles > 0) S.spin = o->spin_limit_cycles;
    KC_TRY(build_tasks(P, S.rpt, A, s, &S.tasks, &S.ntasks_dev, nullptr));
    S.ntasks = tasks_bound(P, S.rpt);
    S.nrhs_cap = nrhs_cap;
    KC_TRY(A.get(&S.cnt, P->N));
    KC_TRY(A.get(&S.acc, S.ntasks * nrhs_cap));
    KC_TRY(A.get(&S.gcnt, S.ntasks));
    KC_TRY(A.get(&S.ticket, 2));
    KC_TRY(A.get(&S.status, 1));
    KC_TRY(A.get(&S.y, P->N * nrhs_cap));
    KC_TRY(A.get(&S.xf, P->N * nrhs_cap));
    return KC_OK;
}

// z = (L L^T)^{-1} rhs, point-major, positions order.  Does not synchronise;
// the status word is checked by solver_check.
template <typename T, int NR>
static kc_status solve_launch(Solver& S, SolveArgs<T> a, int nrhs, cudaStream_t s) {
    constexpr bool PAIR = std::is_same<T, float>::value;
    const kc_pattern* P = S.P;
    // CTAs of 8 warps: as many as fit, and no more than about KC_SOLVE_WAVES
    // warps per row (column chunk) of a dependency level; the rows go out in level
    // order, so further warps would only wait and poll.
    auto launch = [&](void (*kfn)(SolveArgs<T>), int64_t items) -> kc_status {
        int per_sm = 0;
        KC_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kfn, 256, 0));
        const double want = KC_SOLVE_WAVES * (double)items / (double)(P->depth > 0 ? P->depth : 1);
        const int64_t full = (int64_t)sm_count() * (per_sm > 0 ? per_sm : 1);
        const int64_t ctas = (int64_t)(want / 8.0) + 1;
        ::kc::note_launch(), kfn<<<(unsigned)(ctas < full ? ctas : full), 256, 0, s>>>(a);
        KC_CUDA(cudaGetLastError());
        return KC_OK;
    };
    const size_t words = sizeof(unsigned long long) * (size_t)P->N * NR;
    KC_CUDA(cudaMemsetAsync(S.y, 0xff, words, s));  // unset
    KC_CUDA(cudaMemsetAsync(PAIR ? (void*)S.xf : (void*)a.x, 0xff, words, s));
    KC_CUDA(cudaMemsetAsync(S.ticket, 0, 2 * sizeof(unsigned long long), s));
    KC_CUDA(cudaMemsetAsync(S.status, 0, sizeof(int), s));
    KC_CUDA(cudaMemsetAsync(S.cnt, 0, sizeof(unsigned) * P->N, s));
    KC_CUDA(cudaMemsetAsync(S.gcnt, 0, sizeof(unsigned) * S.ntasks, s));
    a.ticket = S.ticket;
    if constexpr (PAIR) KC_TRY(launch(fwd_solve_pair_k<NR>, P->N));
    else KC_TRY(launch(fwd_solve_k<T, NR>, P->N));
    a.ticket = S.ticket + 1;
    if constexpr (PAIR) KC_TRY(launch(bwd_solve_pair_k<NR>, S.ntasks));
    else KC_TRY(launch(bwd_solve_k<T, NR>, S.ntasks));
    return KC_OK;
}

template <typename T>
static SolveArgs<T> solve_args(Solver& S, const T* val, const double* diag, double diag_fallback, const double* rhs,
                               double* z);

// z = (L L^T)^{-1} rhs, point-major with stride nrhs (a power of two <= 16),
// positions order.  Does not synchronise; the status word is checked by
// solver_check.
template <typename T>
kc_status solver_apply(Solver& S, const T* val, const double* diag, double diag_fallback, const double* rhs,
                       double* z, int nrhs, cudaStream_t s) {
    if (nrhs < 1 || nrhs > 16 || (nrhs & (nrhs - 1)) || nrhs > S.nrhs_cap)
        return fail(KC_EINVAL, "internal: solver stride must be a power of two <= 16");
    SolveArgs<T> a = solve_args<T>(S, val, diag, diag_fallback, rhs, z);
    switch (nrhs) {
        case 1: return solve_launch<T, 1>(S, a, nrhs, s);
        case 2: return solve_launch<T, 2>(S, a, nrhs, s);
        case 4: return solve_launch<T, 4>(S, a, nrhs, s);
        case 8: return solve_launch<T, 8>(S, a, nrhs, s);
        default: return solve_launch<T, 16>(S, a, nrhs, s);
    }
}

template <typename T>
static SolveArgs<T> solve_args(Solver& S, const T* val, const double* diag, double diag_fallback, const double* rhs,
                               double* z) {
    const kc_pattern* P = S.P;
    SolveArgs<T> a;
    a.N = P->N;
    a.rowptr = P->rowptr;
    a.col = P->col;
    a.colptr = P->colptr;
    a.rowidx = P->rowidx;
    a.slot = P->slot;
    a.order = P->order;
    a.tasks = S.tasks;
    a.ntasks = S.ntasks_dev;
    a.rpt = S.rpt;
    a.val = val;
    a.diag = diag;
    a.diag_fallback = diag_fallback;
    a.b = rhs;
    a.y = S.y;
    a.x = z;
    a.yf = (float2*)S.y;  // same bytes as the FP64 vector
    a.xf = S.xf;
    a.acc = S.acc;
    a.cnt = S.cnt;
    a.gcnt = S.gcnt;
    a.status = S.status;
    a.spin_limit = S.spin;
    return a;
}
template kc_status solver_apply<double>(Solver&, const double*, const double*, double, const double*, double*, int,
                                        cudaStream_t);
template kc_status solver_apply<float>(Solver&, const float*, const double*, double, const double*, double*, int,
                                       cudaStream_t);

kc_status solver_check(Solver& S, cudaStream_t s) {
    int h = 0;
    KC_CUDA(cudaMemcpyAsync(&h, S.status, sizeof(int), cudaMemcpyDeviceToHost, s));
    KC_CUDA(cudaStreamSynchronize(s));
    if (h == DEV_TIMEOUT) return fail(KC_ETIMEOUT, "solve: a dependency wait ran out");
    if (h != 0) return fail(KC_ECUDA, "solve: device status " + std::to_string(h));
    return KC_OK;
}

// The permutations between original-order right-hand sides b[r*N + i] and
// point-major vectors in position order v[k*stride + r] (perm[k] = i), by
// tiles of 32 points in original order: the rows of b are read and written
// coalesced, and each point's stride values form one line (128 bytes at
// stride 16) written or read whole; the inverse permutation is formed first.
constexpr int PM_WARPS = 8;
// pos starts at -1; an index outside 0..N-1 is ignored, and a point without a
// position is skipped by the tiled kernels (no access outside the arrays for
// a perm that is not a permutation)
__global__ void pm_inverse_perm_k(const int32_t* __restrict__ perm, int64_t N, int32_t* __restrict__ pos) {
    const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (k < N) {
        const int32_t i = perm[k];
        if (i >= 0 && i < N) pos[i] = (int32_t)k;
    }
}
__global__ void __launch_bounds__(PM_WARPS * 32) to_point_major_tiled_k(const double* __restrict__ b,
                                                                       const int32_t* __restrict__ pos, int64_t N,
                                                                       int nrhs, int stride, double* __restrict__ out) {
    __shared__ double tile[PM_WARPS][32][17];
    const int lane = lane_id(), w = threadIdx.x >> 5;
    const int64_t i0 = ((int64_t)blockIdx.x * PM_WARPS + w) * 32;
    if (i0 >= N) return;
    const bool in = i0 + lane < N;
    for (int r = 0; r < stride; ++r) tile[w][lane][r] = (in && r < nrhs) ? b[(int64_t)r * N + i0 + lane] : 0.0;
    __syncwarp();
    for (int e = lane; e < 32 * stride; e += 32) {
        const int p = e / stride, r = e - p * stride;
        const int32_t k = i0 + p < N ? pos[i0 + p] : -1;
        if (k >= 0) out[(int64_t)k * stride + r] = tile[w][p][r];
    }
}
__global__ void __launch_bounds__(PM_WARPS * 32) from_point_major_tiled_k(const double* __restrict__ xp,
                                                                         const int32_t* __restrict__ pos, int64_t N,
                                                                         int nrhs, int stride, double* __restrict__ x) {
    __shared__ double tile[PM_WARPS][32][17];
    const int lane = lane_id(), w = threadIdx.x >> 5;
    const int64_t i0 = ((int64_t)blockIdx.x * PM_WARPS + w) * 32;
    if (i0 >= N) return;
    for (int e = lane; e < 32 * stride; e += 32) {
        const int p = e / stride, r = e - p * stride;
        const int32_t k = i0 + p < N ? pos[i0 + p] : -1;
        tile[w][p][r] = k >= 0 ? xp[(int64_t)k * stride + r] : 0.0;
    }
    __syncwarp();
    if (i0 + lane < N)
        for (int r = 0; r < nrhs; ++r) x[(int64_t)r * N + i0 + lane] = tile[w][lane][r];
}

static kc_status inverse_perm(const int32_t* perm, int64_t N, int32_t** pos, cudaStream_t s) {
    KC_TRY(scratch_alloc((void**)pos, sizeof(int32_t) * (size_t)(N > 0 ? N : 1), s));
    KC_CUDA(cudaMemsetAsync(*pos, 0xFF, sizeof(int32_t) * (size_t)(N > 0 ? N : 1), s));
    ::kc::note_launch(), pm_inverse_perm_k<<<blocks_for(N, 256), 256, 0, s>>>(perm, N, *pos);
    KC_CUDA(cudaGetLastError());
    return KC_OK;
}

kc_status to_point_major(const double* b, const int32_t* perm, int64_t N, int nrhs, double* out, cudaStream_t s,
                         int stride) {
    if (stride < nrhs) stride = nrhs;
    if (stride > 16) {
        ::kc::note_launch(), to_point_major_k<<<blocks_for(N * stride, 256), 256, 0, s>>>(b, perm, N, nrhs, stride, out);
        KC_CUDA(cudaGetLastError());
        return KC_OK;
    }
    int32_t* pos = nullptr;
    KC_TRY(inverse_perm(perm, N, &pos, s));
    ::kc::note_launch(), to_point_major_tiled_k<<<blocks_for(N, PM_WARPS * 32), PM_WARPS * 32, 0, s>>>(b, pos, N, nrhs,
                                                                                                   stride, out);
    const cudaError_t e = cudaGetLastError();
    cudaFreeAsync(pos, s);
    if (e != cudaSuccess) return cuda_fail(e, "to_point_major_tiled_k");
    return KC_OK;
}
kc_status from_point_major(const double* xp, const int32_t* perm, int64_t N, int nrhs, double* x, cudaStream_t s,
                           int stride) {
    if (stride < nrhs) stride = nrhs;
    if (stride > 16) {
        ::kc::note_launch(), from_point_major_k<<<blocks_for(N * nrhs, 256), 256, 0, s>>>(xp, perm, N, nrhs, stride, x);
        KC_CUDA(cudaGetLastError());
        return KC_OK;
    }
    int32_t* pos = nullptr;
    KC_TRY(inverse_perm(perm, N, &pos, s));
    ::kc::note_launch(), from_point_major_tiled_k<<<blocks_for(N, PM_WARPS * 32), PM_WARPS * 32, 0, s>>>(xp, pos, N, nrhs,
                                                                                                     stride, x);
    const cudaError_t e = cudaGetLastError();
    cudaFreeAsync(pos, s);
    if (e != cudaSuccess) return cuda_fail(e, "from_point_major_tiled_k");
    return KC_OK;
}

kc_status solve_impl(const kc_pattern* P, int prec, const void* val, const double* diag, const kc_kernel* kern,
                     const int32_t* perm, const double* b, int nrhs, double* x, const kc_opts* o, cudaStream_t s) {
    KernelParams kp;
    KC_TRY(kernel_params(kern, &kp));
    if (nrhs < 1 || nrhs > 16) return fail(KC_EINVAL, "nrhs must be in 1..16");
    if (prec != KC_FP64 && prec != KC_FP32_FORM) return fail(KC_EINVAL, "prec must be KC_FP64 or KC_FP32_FORM");
    int ns = 1;
    while (ns < nrhs) ns <<= 1;  // padded stride: aligned gathers; the extra columns stay zero
    Arena A(s);
    Solver S;
    KC_TRY(solver_init(S, P, ns, o, A, s));
    double *bp, *zp;
    KC_TRY(A.get(&bp, P->N * ns));
    KC_TRY(A.get(&zp, P->N * ns));
    KC_TRY(to_point_major(b, perm, P->N, nrhs, bp, s, ns));
    double fb = sqrt(kp.sigma2 + kp.nugget);
    if (prec == KC_FP64) KC_TRY(solver_apply<double>(S, (const double*)val, diag, fb, bp, zp, ns, s));
    else KC_TRY(solver_apply<float>(S, (const float*)val, diag, fb, bp, zp, ns, s));
    KC_TRY(from_point_major(zp, perm, P->N, nrhs, x, s, ns));
    return solver_check(S, s);
}

}  // namespace kc
