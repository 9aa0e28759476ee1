// a2: the maximin ordering (Section 2.3), exact, on the device.
//
// Definition (greedy): the first point is original index 0; each next point
// is the unselected point with the largest squared distance v(p) to the
// selected set, ties to the smaller original index; l = sqrt(v at selection).
// Write key(p) = (v(p), -index).  The l values are non-increasing, so the
// order is the sort of the points by final key, and each point's final v is
// what must be found.
//
// Parallel rounds.  Keep for every undecided point its v over the points
// selected so far.  An undecided point q is *dominant* when no undecided
// point of larger key lies at squared distance < v(q).  Then v(q) is final:
// no point that ends up before q can come closer than v(q) -- the first such
// point would have to be selected while q, of larger key, is still
// available.  All dominant points of a round are selected together.  A
// selected p then lowers v(q) := min(v(q), d2(p,q)) for undecided q of
// smaller key; undecided q of larger key are left alone, which is exact: q
// was within reach of p only if d2(p,q) >= v(p), and if q later falls below
// p its value is already below d2(p,q).
//
// Rounds run in bands of keys: with vmax the largest undecided v, the band
// holds the undecided points with v >= KC_ORDER_BAND vmax; only band points can dominate
// band points, so the dominance search uses a grid of band points with cells of
// a quarter of sqrt(vmax) (more where the points are too few for that), whose
// largest points alone are searched for where a cell holds several.  The updates
// scan a fixed fine grid of all points.  All bands run in one cooperative launch.
// Finally the points are sorted by (v descending, index ascending).
//
// Bound by latency: about 50 rounds of dependent scans, each between grid
// barriers.  Measured (before: a dozen launches and two waits of the host per
// round): 2^20 points of a jittered grid 16.0 -> 8.4 ms, 250,007 points of a
// swiss roll in R^20 22.4 -> 15.3 (34 in a process that has used many streams,
// where every launch costs more), 131,071 points of the cube 13.3 -> 7.6, 100,003
// in the square 9.2 -> 3.7, 2000 4.6 -> 1.2; 60,000 points of the cube in R^20 320 ->
// 260, 100,003 in R^8 154 -> 153, 5000 in R^20 16.1 -> 10.6; 100,000 points with heavy
// tails (most of them in a few cells) 1170 -> 1155.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>

#include "grid.cuh"

namespace kc {

// out[q] = rows ids[q] of the n x w array a
__global__ void gather_rows_k(const double* __restrict__ a, int w, const int32_t* __restrict__ ids, int64_t n,
                              double* __restrict__ out) {
    const int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (q < n)
        for (int t = 0; t < w; ++t) out[q * w + t] = a[(int64_t)ids[q] * w + t];
}

// Floats of a point's row of the float copy: past three axes rows are filled up
// with zeros to whole 16 bytes, so that a screen reads them by 16-byte loads
// (a warp's 32 rows by single floats take a trip to L1 per float and line).
__host__ __device__ __forceinline__ int row_floats(int d) { return d <= 3 ? d : (d + 3) & ~3; }
// screen_f32 on such rows (HIGH: d > 3): the same sum (the filling adds zeros) and decision
template <bool HIGH>
__device__ __forceinline__ int screen_rows(const float* a, const float* b, int d, float Rf, float delta) {
    if constexpr (!HIGH) return screen_f32(a, b, d, Rf, delta);
    float s = 0.f;
    for (int t = 0; t < d; t += 4) {
        const float4 u = *(const float4*)(a + t), v = *(const float4*)(b + t);
        const float w0 = u.x - v.x, w1 = u.y - v.y, w2 = u.z - v.z, w3 = u.w - v.w;
        s = fmaf(w3, w3, fmaf(w2, w2, fmaf(w1, w1, fmaf(w0, w0, s))));
    }
    const float dist = sqrtf(s);
    const float M = sqrtf((float)d) * delta + (float)(d + 6) * 1.1920929e-7f * fmaxf(dist, Rf);
    if (dist - M > Rf) return 0;
    if (dist + M < Rf) return 1;
    return -1;
}

// state in grid order (gpos): coordinates xg, original index idg, v2, stat
__global__ void ord_init_k(const double* __restrict__ x, int d, const int32_t* __restrict__ gsorted, int64_t N,
                           double* __restrict__ xg, int32_t* __restrict__ idg, double* __restrict__ v2,
                           int* __restrict__ stat, Origin org, float* __restrict__ xgf) {
    int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= N) return;
    int64_t id = gsorted[q];
    const int df = row_floats(d);
    for (int t = 0; t < d; ++t) {
        xg[q * d + t] = x[id * d + t];
        xgf[q * df + t] = (float)(x[id * d + t] - org.lo[t]);
    }
    for (int t = d; t < df; ++t) xgf[q * df + t] = 0.f;
    idg[q] = (int32_t)id;
    if (id == 0) {
        v2[q] = INFINITY;
        stat[q] = 1;
    } else {
        v2[q] = dist2_exact(x + id * d, x, d);
        stat[q] = 0;
    }
}

// Keys compare on the bit patterns of the squared distances: for v >= 0
// (and +inf) IEEE doubles order like their bits as integers, and integer
// compares stay off the GB300's small FP64 pipe.
__device__ __forceinline__ long long vbits(double v) { return __double_as_longlong(v); }
__device__ __forceinline__ bool key_above(double va, int ia, double vb, int ib) {
    const long long a = vbits(va), b = vbits(vb);
    return a > b || (a == b && ia < ib);
}

#ifndef KC_DOM_BUDGET
#define KC_DOM_BUDGET 32
#endif
constexpr int DOM_THREAD_BUDGET = KC_DOM_BUDGET;
// Candidates of the first look of points in more than three dimensions (below).
constexpr int LIST_BUDGET = 16;

// What the band rounds read and write.  v2 and stat change between the phases of
// one launch: they go without __restrict__, so that they are never read through
// the non-coherent path.
struct BandArgs {
    int64_t N;
    int d, gs, df;                      // df: floats of a row of xgf
    Grid g0;                            // fine grid of all points
    const int64_t* __restrict__ cstart;  // its cells
    const double* __restrict__ xg;      // coordinates in grid order
    const float* __restrict__ xgf;      // float copy minus the box corner
    const double* __restrict__ gxg;     // grid coordinates (stride gs)
    const int4* __restrict__ pcell;     // a point's cell on the fine grid
    const int32_t* __restrict__ idg;
    float delta;
    double* v2;
    int* stat;
    int32_t *blist, *bcell, *bsorted, *bcnt, *bstart, *hard, *sel;
    long long* cmax;
    int32_t* champ;                     // the cell's undecided point of largest key (dense bands)
    int32_t* wit;                       // a point that dominated it, -1: none yet
    double* wd;                         // and its squared distance
    int* part;                          // scan: one sum per block
    struct BandCtl* ctl;
    unsigned* flags;  // of the grid barrier
    double lo[3], hi[3];
    long long limit;
    int beat_shift;
};
// Counters: of a band by its parity, of a round modulo 3 (reset two phases before their next use).
struct BandCtl {
    unsigned long long vmax[2];
    unsigned open[2], nb[2], occ[2];
    unsigned nsel[3], nact[3], nhard[3], nlong[3];
    unsigned bar, beat;
    int status, rounds;
};
// A warp's sign of work, where an item or a long part of one begins: at most once per
// 2^beat_shift cycles, a 16th of the limit or less.
__device__ __forceinline__ void beat(const BandArgs& A) {
    __shared__ unsigned last[8];
    const unsigned t = (unsigned)(clock64() >> A.beat_shift);
    volatile unsigned* mine = &last[threadIdx.x >> 5];
    if (*mine != t) {
        *mine = t;
        atomicAdd(&A.ctl->beat, 1u);
    }
}

// Band grid: cells a quarter of the largest search radius, at most about 2 nb of
// them (any grid gives the same order).
__device__ __noinline__ void band_grid(const BandArgs& A, double vmax, int64_t nb, Grid& g) {
    g.dg = A.g0.dg;
    g.c = g.inv_c = 1.0;
    g.n[0] = g.n[1] = g.n[2] = 1;
    g.ncells = 1;
    double vol = 1.0, emax = 0.0, ext[3] = {0.0, 0.0, 0.0};
    int nz = 0;
    for (int t = 0; t < g.dg; ++t) {
        g.lo[t] = A.lo[t];
        ext[t] = A.hi[t] > A.lo[t] ? A.hi[t] - A.lo[t] : 0.0;
        if (ext[t] > 0.0) {
            vol *= ext[t];
            ++nz;
        }
        emax = fmax(emax, ext[t]);
    }
    if (!(emax > 0.0)) return;
    if (!(emax > 1e-290 && emax < 1e300)) {
        one_cell(g);
        return;
    }
    const int64_t most = 2 * nb + 1;
    const double q = vol / (double)most;
    double c = nz == 1 ? q : nz == 2 ? sqrt(q) : cbrt(q);
    c = fmax(c, 0.25 * sqrt(vmax));
    for (int step = 0; step < 4096; ++step) {
        int64_t tot = 1;
        bool fits = c > 0.0;
        for (int t = 0; t < g.dg && fits; ++t) {
            const double f = floor(ext[t] / c) + 1.0;
            if (!(f <= 1e6)) fits = false;
            else {
                g.n[t] = (int)f;
                tot *= g.n[t];
                fits = tot <= most;
            }
        }
        if (fits) {
            g.ncells = tot;
            g.c = c;
            g.inv_c = 1.0 / c;
            return;
        }
        c = c > 0.0 ? c * 1.25 : emax * 1e-6;
    }
    one_cell(g);
}

// Cells to either side of a point's own that cover sqrt(v) on the grid g, by FP32
// arithmetic with slack (a larger box is as good) where float holds v.
__device__ __forceinline__ int span_of_v(const Grid& g, double v, float inv_c, int t) {
    if (!(v > 1e-30 && v < 1e30 && inv_c > 1e-30f && inv_c < 1e30f)) return span_for(g, sqrt(v), t);
    const float f = sqrtf((float)v) * inv_c * (1.0f + 1e-5f) + 1e-5f;
    return f > (float)g.n[t] ? g.n[t] : min(g.n[t], (int)f + 1);
}

// Does the undecided band point p dominate q (larger key, closer than sqrt(vq))?
// Its squared distance if it does, else infinity.
template <bool HIGH>
__device__ __forceinline__ double dominates(const BandArgs& A, int p, int q, double vq, float rq, int idq) {
    if (p == q || A.stat[p] != 0) return INFINITY;
    if (!key_above(A.v2[p], A.idg[p], vq, idq)) return INFINITY;
    if (screen_rows<HIGH>(A.xgf + (int64_t)p * A.df, A.xgf + (int64_t)q * A.df, A.d, rq, A.delta) == 0) return INFINITY;
    const double dd = dist2_exact(A.xg + (int64_t)p * A.d, A.xg + (int64_t)q * A.d, A.d);
    return dd < vq ? dd : INFINITY;
}

// A point that dominates the undecided band point q, with its squared distance
// in wd; -1: none, q is dominant.  One thread scans the band grid ring by ring
// outward from q's cell: most points meet a dominator within the first rings
// (ring r holds no point closer than (r-1) cells).  It gives up (-2) when the
// scan would go past DOM_THREAD_BUDGET candidates: an undominated point has to look at every band point within sqrt(v), which is a
// warp's work.
template <bool HIGH>
__device__ __forceinline__ int dominator_thread(const BandArgs& A, const Grid& gb, int q, double vq, int budget,
                                                double& wd) {
    const long long bq = vbits(vq);
    const float rq = sqrtf((float)vq);
    const int idq = A.idg[q];
    const double R = sqrt(vq);
    const int dg = gb.dg;
    int c[3] = {0, 0, 0};
    int maxr = 0;
    for (int t = 0; t < dg; ++t) {
        c[t] = cell_coord(gb, A.gxg[(int64_t)q * A.gs + t], t);
        maxr = max(maxr, span_for(gb, R, t));
    }
    for (int r = 0; r <= maxr; ++r) {
        if (r >= 2 && (double)(r - 1) * gb.c > R) break;
        const int z0 = dg > 2 ? max(0, c[2] - r) : 0, z1 = dg > 2 ? min(gb.n[2] - 1, c[2] + r) : 0;
        const int y0 = dg > 1 ? max(0, c[1] - r) : 0, y1 = dg > 1 ? min(gb.n[1] - 1, c[1] + r) : 0;
        for (int cz = z0; cz <= z1; ++cz)
            for (int cy = y0; cy <= y1; ++cy) {
                // the cells of this ring in the row: all of [c-r, c+r] on an edge row, else the two ends
                const bool edge = r == 0 || (dg > 2 && abs(cz - c[2]) == r) || (dg > 1 && abs(cy - c[1]) == r);
                const int64_t base = ((int64_t)cz * gb.n[1] + cy) * gb.n[0];
                const int step = edge ? 1 : 2 * r;
                for (int cx = c[0] - r; cx <= c[0] + r; cx += step) {
                    if (cx < 0 || cx >= gb.n[0]) continue;
                    if (A.cmax[base + cx] < bq) continue;  // no larger key in this cell
                    const int f0 = A.bstart[base + cx], f1 = A.bstart[base + cx + 1];
                    if (f1 - f0 > budget) return -2;
                    budget -= f1 - f0;
                    for (int f = f0; f < f1; ++f) {
                        const int p = A.bsorted[f];
                        const double dd = dominates<HIGH>(A, p, q, vq, rq, idq);
                        if (dd < vq) {
                            wd = dd;
                            return p;
                        }
                    }
                }
            }
    }
    return -1;
}

// Lane whose range [inc - len, inc) holds m, from the inclusive sums inc of the lanes' lengths
// (m past the last: any lane).
__device__ __forceinline__ int which_row(int inc, int m) {
    int row = 0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
        if (__shfl_sync(0xffffffffu, inc, row + o - 1) <= m) row += o;
    return row;
}

// The same by a warp, a lane per cell of the box around q.  (With the warp on
// one cell at a time the cells of a box were a chain of dependent loads.)
template <bool HIGH, bool DENSE>
__device__ __forceinline__ int dominator_warp(const BandArgs& A, const Grid& gb, int q, double vq, double& wd) {
    constexpr int SCAN = 4;
    const unsigned FULL = 0xffffffffu;
    const int lane = lane_id();
    const long long bq = vbits(vq);
    const float rq = sqrtf((float)vq);
    const int idq = A.idg[q];
    const double R = sqrt(vq);
    int lo[3] = {0, 0, 0}, n[3] = {1, 1, 1};
    for (int t = 0; t < gb.dg; ++t) {
        const int c = cell_coord(gb, A.gxg[(int64_t)q * A.gs + t], t), sp = span_for(gb, R, t);
        lo[t] = max(0, c - sp);
        n[t] = min(gb.n[t] - 1, c + sp) - lo[t] + 1;
    }
    const int cells = n[0] * n[1] * n[2];
    int own = 0;
    if constexpr (HIGH)
        for (int t = gb.dg - 1; t >= 0; --t) own = own * n[t] + cell_coord(gb, A.gxg[(int64_t)q * A.gs + t], t) - lo[t];
    auto cell_at = [&](int t) {
        const int row = t / n[0];
        return ((int64_t)(lo[2] + row / n[1]) * gb.n[1] + lo[1] + row % n[1]) * gb.n[0] + lo[0] + t % n[0];
    };
    if constexpr (DENSE) {  // the cells' largest points first: they dominate nearly whatever is dominated
        for (int t0 = 0; t0 < cells; t0 += 32) {
            int p = -1;
            double dd = INFINITY;
            if (t0 + lane < cells) {
                const int64_t cell = cell_at(t0 + lane);
                if (A.cmax[cell] >= bq) {
                    p = A.champ[cell];  // there is one: its value is at least vq, so at least T
                    dd = dominates<HIGH>(A, p, q, vq, rq, idq);
                }
            }
            const unsigned hits = __ballot_sync(FULL, dd < vq);
            if (hits) {
                wd = __shfl_sync(FULL, dd, __ffs(hits) - 1);
                return __shfl_sync(FULL, p, __ffs(hits) - 1);
            }
        }
    }
    // then all points of the cells with a larger key, batches of 32 cells: their
    // points go to the lanes in one sequence, four at a time so that their loads overlap
    for (int t0 = 0; t0 < cells; t0 += 32) {
        int f0 = 0, len = 0;
        if (t0 + lane < cells) {
            const int t = t0 + lane + own;
            const int64_t cell = cell_at(t < cells ? t : t - cells);
            if (A.cmax[cell] >= bq) {
                f0 = A.bstart[cell];
                len = A.bstart[cell + 1] - f0;
            }
        }
        int inc = len;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int up = __shfl_up_sync(FULL, inc, o);
            if (lane >= o) inc += up;
        }
        const int total = __shfl_sync(FULL, inc, 31);
        for (int m0 = 0; m0 < total; m0 += 32 * SCAN) {
            if (lane == 0 && (m0 & 2047) == 2048 - 32 * SCAN) beat(A);
            int p[SCAN];
#pragma unroll
            for (int u = 0; u < SCAN; ++u) {
                const int m = m0 + 32 * u + lane;
                const int row = which_row(inc, m);
                const int f = __shfl_sync(FULL, f0, row) + m - __shfl_sync(FULL, inc - len, row);
                p[u] = m < total ? A.bsorted[f] : -1;
            }
            double v[SCAN];
            int st[SCAN];
#pragma unroll
            for (int u = 0; u < SCAN; ++u) {
                st[u] = p[u] >= 0 ? A.stat[p[u]] : 1;
                v[u] = p[u] >= 0 ? A.v2[p[u]] : 0.0;
            }
            double dd = INFINITY;
            int hit = -1;
#pragma unroll
            for (int u = 0; u < SCAN; ++u)
                if (hit < 0 && st[u] == 0 && vbits(v[u]) >= bq) {
                    dd = dominates<HIGH>(A, p[u], q, vq, rq, idq);
                    if (dd < vq) hit = p[u];
                }
            const unsigned hits = __ballot_sync(FULL, hit >= 0);
            if (hits) {
                wd = __shfl_sync(FULL, dd, __ffs(hits) - 1);
                return __shfl_sync(FULL, hit, __ffs(hits) - 1);
            }
        }
    }
    return -1;
}

// one slot of a list per calling thread, by one atomic per group of threads
__device__ __forceinline__ unsigned list_slot(unsigned* n) {
    const unsigned m = __activemask();
    const int leader = __ffs(m) - 1;
    unsigned base = 0;
    if (lane_id() == leader) base = atomicAdd(n, (unsigned)__popc(m));
    return __shfl_sync(m, base, leader) + __popc(m & ((1u << lane_id()) - 1u));
}

// ---- greedy steps for the coarsest points: each step selects the argmax of
// the previous step's per-block candidates and pushes it to the points near it.
// 64, 96, 128, 256 and 512 of them: 10.1, 9.0, 9.0, 9.35 and 9.5 ms for the ordering
// of 2^20 points, 3.52, 3.53, 3.49, 3.70 and 4.0 for the path of 2000 (all at a
// band of 0.25; at 0.16 and 128 steps 8.8 and 3.43, at 0.4 9.0 and 3.75).
constexpr int GREEDY_THREADS = 1024;
#ifndef KC_GREEDY_STEPS
#define KC_GREEDY_STEPS 128
#endif
constexpr int64_t GREEDY_STEPS = KC_GREEDY_STEPS;  // coarsest points selected one at a time
// Where a twentieth of the variance lies outside the grid's three axes (a cube of
// four dimensions has a quarter there, a noisy sheet next to nothing), the grid
// prunes little and the first rounds look at nearly all pairs: more steps then.
// 128, 512, 1024 and 2048 of them: 160, 149, 141 and 124 ms for 100,003 points of
// the cube in R^8, 11.8, 10.8, 12.2 and 16.5 for 5000 in R^20, 18.5, 14.6, 14.7 and
// 17.5 for 100,003 in R^4; 15.7, 17.6, 19.9 and 26.3 for 250,007 of a swiss roll.
constexpr int64_t GREEDY_STEPS_SPREAD = 512;
// A band holds the undecided points with v >= KC_ORDER_BAND * (largest v).
#ifndef KC_ORDER_BAND
#define KC_ORDER_BAND 0.16
#endif

// the better of two candidates (v2 desc, original index asc; g < 0: none)
struct Cand {
    double v;
    int i, g;
    __device__ __forceinline__ void take(double vo, int io, int go) {
        if (go >= 0 && (g < 0 || key_above(vo, io, v, i))) {
            v = vo;
            i = io;
            g = go;
        }
    }
    __device__ __forceinline__ void warp_best() { best_of<16>(); }
    template <int FROM>
    __device__ __forceinline__ void best_of() {
#pragma unroll
        for (int o = FROM; o > 0; o >>= 1)
            take(__shfl_xor_sync(0xffffffffu, v, o), __shfl_xor_sync(0xffffffffu, i, o), __shfl_xor_sync(0xffffffffu, g, o));
    }
};
// A grid-wide barrier for a cooperative launch (every block resident).  Blocks
// arrive at one counter, which only grows; the last of a phase tells every block
// at a word in a sector of its own (a single word that all poll was slower:
// 10.6 against 9.35 ms for the ordering of 2^20 points, 25.4 against 24.6 for
// the 250,007 of a swiss roll).  A wait ends, with the status word set and false
// returned, when no warp has given a sign of work (`beat`) for `limit` cycles, or
// another block has failed: how long a phase's scans take depends on the points, so
// a limit on the wait itself would refuse large sets that the grid prunes little.
// `phase`: the barriers passed so far, kept by the caller (all threads).
constexpr int BAR_STRIDE = 8;  // words between the blocks' flags
__device__ bool grid_barrier(unsigned* count, unsigned* flags, unsigned& phase, int* status, const unsigned* beat,
                             long long limit) {
    __shared__ int ok, last;
    __syncthreads();
    ++phase;
    if (threadIdx.x == 0) {
        ok = 1;
        fence_acq_rel_gpu();  // this block's writes before its arrival
        last = atomicAdd(count, 1u) == phase * gridDim.x - 1u;
        fence_acq_rel_gpu();  // acquire (the last block): the others' writes
    }
    __syncthreads();
    if (last) {
        for (unsigned b = threadIdx.x; b < gridDim.x; b += blockDim.x)
            asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(flags + b * BAR_STRIDE), "r"(phase) : "memory");
    } else if (threadIdx.x == 0) {
        const unsigned* mine = flags + blockIdx.x * BAR_STRIDE;
        long long t0 = clock64();
        unsigned seen = 0;
        for (int poll = 1; ld_acquire_u32(mine) != phase; ++poll) {
            bool stop = (poll & 63) == 0 && ld_volatile_s32(status) != 0;
            if (clock64() - t0 > limit) {
                const unsigned now = *(const volatile unsigned*)beat;
                stop |= now == seen;
                seen = now;
                t0 = clock64();
            }
            if (stop) {
                atomicCAS(status, 0, DEV_TIMEOUT);
                ok = 0;
                break;
            }
            if (poll > 8) __nanosleep(32);
        }
        fence_acq_rel_gpu();  // acquire: the other blocks' writes
    }
    __syncthreads();
    return ok != 0;
}

// A greedy step's candidates: the squared distance as its bits, which order like
// the values (integer compares: the FP64 pipe takes 16 clocks for a warp's
// compare), the point's original index and its place (g < 0: none).
struct GreedyCand {
    unsigned long long v;
    int i, g;
};
__device__ __forceinline__ GreedyCand no_cand() { return GreedyCand{0ull, INT_MAX, -1}; }
__device__ __forceinline__ void greedy_take(GreedyCand& c, unsigned long long v, int i, int g) {
    if (v > c.v || (v == c.v && i < c.i)) c = GreedyCand{v, i, g};
}
// the best of the warp's candidates (largest v, then smallest i), in every lane
__device__ __forceinline__ GreedyCand greedy_best(const GreedyCand& c) {
    const unsigned FULL = 0xffffffffu;
    const unsigned hi = (unsigned)(c.v >> 32), mh = __reduce_max_sync(FULL, hi);
    const unsigned lo = hi == mh ? (unsigned)c.v : 0u, ml = __reduce_max_sync(FULL, lo);
    const bool top = hi == mh && lo == ml;
    const int mi = __reduce_min_sync(FULL, top ? c.i : INT_MAX);
    const int src = __ffs(__ballot_sync(FULL, top && c.i == mi)) - 1;
    return GreedyCand{(unsigned long long)mh << 32 | ml, mi, __shfl_sync(FULL, c.g, src)};
}
// a nonnegative double's bits as a float, rounded down (integer operations), but
// not below float's smallest normal number
__device__ __forceinline__ float float_below(unsigned long long v) {
    const unsigned h = (unsigned)(v >> 32);
    if (h < 897u << 20) return 1.1754944e-38f;
    if (h >= 1151u << 20) return h >= 2047u << 20 ? INFINITY : 3.4028234e38f;
    return __uint_as_float(((h - (896u << 20)) << 3) | ((unsigned)v >> 29));
}

// All greedy steps in one cooperative launch of at most one CTA per SM.  The points
// lie in cell order, so stretches of 32 (or a small multiple) have small boxes; a
// warp has up to 32 of them, the state of each, its box and its best candidate, in
// a lane.  A step looks at a stretch's points only if the winner is one of them or
// its distance from the box is not above the largest of their values, for
// otherwise none can change.  Neighbouring stretches go to different blocks and
// warps: a step takes as long as the warp with the most to look at, whose chains
// of loads follow one another, and so a winner's surroundings are spread over all
// the SMs.  Every block sends the best of its warps to a slot in every block's row
// of buffer k & 1 and reads its own row, so every block finds the same winner
// (with one slot a block that all poll, the polls crowd a few lines: 8.9 us a step).  The slots carry
// their own readiness, a parity bit in each of their two words that changes with
// every use of a buffer: no barrier and no fence.  A block writes a buffer again
// only after it has read the next one whole, which the others write after they
// have read this one.  The shared buffers alternate likewise: a warp writes one
// again only after a block barrier that every warp reaches past its last read.
// A step took 14.6 us at 2^20 points and 7.4 at 2000 with a grid barrier and 608
// blocks, 10.9 and 3.1 with the slots but every point looked at and FP64
// compares, and 4.8 and 2.1 now.
template <bool HIGH>
__global__ void __launch_bounds__(GREEDY_THREADS, 1)
    ord_greedy_loop_k(const double* __restrict__ xg, int d, const int32_t* __restrict__ idg, double* v2, int* stat,
                      int64_t N, int64_t steps, ulonglong2* slots, const float* __restrict__ xgf, float delta,
                      int* status, long long limit) {
    __shared__ GreedyCand sh[2][32], sx[2][32];
    const int nblk = gridDim.x, lane = lane_id(), wrp = threadIdx.x >> 5;
    const unsigned FULL = 0xffffffffu;
    const unsigned long long PB = 1ull << 63;
    const int64_t nw = (int64_t)nblk * (GREEDY_THREADS / 32);
    // stretches of `per` points; lane j keeps the state of the warp's stretch j
    const int64_t per = 32 * ((N + 1024 * nw - 1) / (1024 * nw)), ns = (N + per - 1) / per;
    const int64_t gw = (int64_t)wrp * nblk + blockIdx.x;
    const int mine = ns > gw ? (int)((ns - gw + nw - 1) / nw) : 0;  // the warp's stretches, at most 32
    const int da = min(d, 3), df = row_floats(d);
    float lo[3] = {INFINITY, INFINITY, INFINITY}, hi[3] = {-INFINITY, -INFINITY, -INFINITY};  // box, first three axes
    for (int j = 0; j < mine; ++j) {
        const int64_t q0 = (gw + j * nw) * per, q1 = min(N, q0 + per);
#pragma unroll
        for (int t = 0; t < 3; ++t)
            if (t < da) {
                float a = INFINITY, b = -INFINITY;
                for (int64_t q = q0 + lane; q < q1; q += 32) {
                    const float u = xgf[q * df + t];
                    a = fminf(a, u);
                    b = fmaxf(b, u);
                }
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) {
                    a = fminf(a, __shfl_xor_sync(FULL, a, o));
                    b = fmaxf(b, __shfl_xor_sync(FULL, b, o));
                }
                if (lane == j) {
                    lo[t] = a;
                    hi[t] = b;
                }
            }
    }
    const int64_t own = (gw + lane * nw) * per;  // the lane's stretch
    GreedyCand best = no_cand();                 // of the lane's stretch
    float reach = 0.f;                           // not below the largest value of the lane's stretch
    int64_t w = -1;                              // the winner of the previous step
    for (int64_t k = 0; k <= steps; ++k) {
        bool look = lane < mine;
        if (look && w >= 0 && (w < own || w >= own + per)) {
            float s = 0.f;  // not above the squared distance of the winner from the box
#pragma unroll
            for (int t = 0; t < 3; ++t)
                if (t < da) {
                    const float u = xgf[w * df + t];
                    const float g = fmaxf(lo[t] - u, u - hi[t]) * (1.f - 1e-6f) - delta;
                    if (g > 0.f) s = fmaf(g, g, s);
                }
            look = !(s * (1.f - 1e-5f) > reach);
        }
        for (unsigned todo = __ballot_sync(FULL, look); todo; todo &= todo - 1) {
            const int j = __ffs(todo) - 1;
            const int64_t q0 = (gw + j * nw) * per, q1 = min(N, q0 + per);
            GreedyCand c = no_cand();
            for (int64_t q = q0 + lane; q < q1; q += 32) {
                unsigned long long vq = (unsigned long long)__double_as_longlong(v2[q]);
                const int at = idg[q];
                if (q == w) stat[q] = 1;  // v2[w] keeps its final value l^2
                if (q == w || stat[q] != 0) continue;
                if (w >= 0 && screen_rows<HIGH>(xgf + q * df, xgf + w * df, d, sqrtf(float_below(vq)), delta) != 0) {
                    const double dd = dist2_exact(xg + q * d, xg + w * d, d);
                    const unsigned long long u = (unsigned long long)__double_as_longlong(dd);
                    if (u < vq) {
                        vq = u;
                        v2[q] = dd;
                    }
                }
                greedy_take(c, vq, at, (int)q);
            }
            c = greedy_best(c);
            if (lane == j) {
                best = c;
                reach = __uint_as_float(__float_as_uint(float_below(c.v)) + (c.v < 0x7ff0000000000000ull));
            }
        }
        if (k == steps) break;
        {
            const GreedyCand c = greedy_best(best);
            if (lane == 0) sh[k & 1][wrp] = c;
        }
        __syncthreads();
        GreedyCand c = greedy_best(sh[k & 1][lane]);
        if (nblk > 1) {
            ulonglong2* buf = slots + (k & 1) * nblk * nblk;
            const unsigned long long par = ((k >> 1) & 1) ? 0ull : PB;
            if (threadIdx.x < nblk) {
                ulonglong2* to = buf + threadIdx.x * nblk + blockIdx.x;
                // squared distances have no sign bit, indices are below 2^31; no candidate: all ones below it
                const unsigned long long a = c.v | par;
                const unsigned long long b = ((unsigned long long)(unsigned)c.i << 32 | (unsigned)c.g) | par;
                asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};" ::"l"(to), "l"(a), "l"(b) : "memory");
            }
            bool fine = true;
            if (32 * wrp < nblk) {
                c = no_cand();
                const int b = threadIdx.x;
                if (b < nblk) {
                    unsigned long long u, v;
                    const long long t0 = clock64();
                    for (int poll = 1;; ++poll) {
                        asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];"
                                     : "=l"(u), "=l"(v)
                                     : "l"(&buf[blockIdx.x * nblk + b])
                                     : "memory");
                        if ((u & PB) == par && (v & PB) == par) break;
                        if (clock64() - t0 > limit || ((poll & 63) == 0 && ld_volatile_s32(status) != 0)) {
                            atomicCAS(status, 0, DEV_TIMEOUT);
                            fine = false;
                            break;
                        }
                    }
                    c = GreedyCand{u & ~PB, (int)((v & ~PB) >> 32), (int)(unsigned)v};
                }
                c = greedy_best(c);
            }
            if (lane == 0) sx[k & 1][wrp] = 32 * wrp < nblk ? c : no_cand();
            if (__syncthreads_or(!fine)) return;
            c = greedy_best(sx[k & 1][lane]);
        }
        w = c.g;
    }
}

// All bands and their rounds in one cooperative launch, a grid barrier between
// the phases: the host waits once, where it used to wait three times per band
// and twice per round, around a dozen launches each.
//
// HIGH: more than three dimensions.  (Registers for three blocks an SM without most of
// the spills: 329.8 against 305.0 ms for 60,000 points of the cube in R^20.)
template <bool HIGH>
__global__ void __launch_bounds__(256, 4) ord_bands_k(BandArgs A) {
    __shared__ int wsum[8];
    __shared__ int carry;
    __shared__ int active;
    __shared__ Grid gb;  // of the band
    BandCtl* C = A.ctl;
    const float inv_c0 = (float)A.g0.inv_c;
    const int64_t tid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, nt = (int64_t)gridDim.x * blockDim.x;
    const int lane = lane_id();
    const int64_t warp = tid >> 5, nw = nt >> 5;
    const bool first = tid == 0;
    unsigned phase = 0;
    auto barrier = [&]() { return grid_barrier(&C->bar, A.flags, phase, &C->status, &C->beat, A.limit); };
    int round = 0;
    for (int band = 0;; ++band) {
        const int bp = band & 1;
        // largest undecided value, and whether there is any
        {
            unsigned long long m = 0;
            bool any = false;
            for (int64_t q = tid; q < A.N; q += nt)
                if (A.stat[q] == 0) {
                    m = max(m, (unsigned long long)__double_as_longlong(A.v2[q]));
                    any = true;
                }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
            any = __any_sync(0xffffffffu, any);
            if (lane == 0 && any) {
                atomicMax(&C->vmax[bp], m);
                C->open[bp] = 1u;
            }
        }
        if (!barrier()) return;
        if (*(volatile unsigned*)&C->open[bp] == 0u) return;  // every point is decided
        const double vmax = __longlong_as_double((long long)*(volatile unsigned long long*)&C->vmax[bp]);
        const double T = vmax * KC_ORDER_BAND;
        if (first) {
            C->vmax[bp ^ 1] = 0ull;
            C->open[bp ^ 1] = C->nb[bp ^ 1] = C->occ[bp ^ 1] = 0u;
        }
        for (int64_t q = tid; q < A.N; q += nt)
            if (A.stat[q] == 0 && A.v2[q] >= T) A.blist[list_slot(&C->nb[bp])] = (int32_t)q;
        if (!barrier()) return;
        // the band's points by cells: counts, their scan, fill
        const int64_t nb = *(volatile unsigned*)&C->nb[bp];
        if (threadIdx.x == 0) band_grid(A, vmax, nb, gb);
        __syncthreads();
        for (int64_t c = tid; c < gb.ncells; c += nt) A.bcnt[c] = 0;
        if (!barrier()) return;
        for (int64_t e = tid; e < nb; e += nt) {
            const int c = (int)cell_of(gb, A.gxg + (int64_t)A.blist[e] * A.gs);
            A.bcell[e] = c;
            if (atomicAdd(&A.bcnt[c], 1) == 0) list_slot(&C->occ[bp]);
        }
        if (!barrier()) return;
        const int64_t per = ((gb.ncells + gridDim.x - 1) / gridDim.x + 255) / 256 * 256;
        const int64_t c0 = min(gb.ncells, (int64_t)blockIdx.x * per), c1 = min(gb.ncells, c0 + per);
        {
            int sum = 0;
            for (int64_t c = c0 + threadIdx.x; c < c1; c += blockDim.x) sum += A.bcnt[c];
            sum = warp_sum(sum);
            if (lane == 0) wsum[threadIdx.x >> 5] = sum;
            __syncthreads();
            if (threadIdx.x == 0) {
                int t = 0;
                for (int w = 0; w < 8; ++w) t += wsum[w];
                A.part[blockIdx.x] = t;
            }
        }
        if (!barrier()) return;
        {
            int sum = 0;  // the cells before the block's
            for (int b = threadIdx.x; b < (int)blockIdx.x; b += blockDim.x) sum += A.part[b];
            sum = warp_sum(sum);
            if (lane == 0) wsum[threadIdx.x >> 5] = sum;
            __syncthreads();
            if (threadIdx.x == 0) {
                int t = 0;
                for (int w = 0; w < 8; ++w) t += wsum[w];
                carry = t;
            }
            __syncthreads();
            for (int64_t cb = c0; cb < c1; cb += blockDim.x) {
                const int64_t c = cb + threadIdx.x;
                const int n = c < c1 ? A.bcnt[c] : 0;
                int inc = n;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int up = __shfl_up_sync(0xffffffffu, inc, o);
                    if (lane >= o) inc += up;
                }
                if (lane == 31) wsum[threadIdx.x >> 5] = inc;
                __syncthreads();
                int before = carry;
                for (int w = 0; w < (int)(threadIdx.x >> 5); ++w) before += wsum[w];
                if (c < c1) {
                    A.bstart[c] = before + inc - n;
                    A.bcnt[c] = before + inc - n;  // where the cell's next point goes
                }
                __syncthreads();
                if (threadIdx.x == blockDim.x - 1) carry = before + inc;
                __syncthreads();
            }
            if (first) A.bstart[gb.ncells] = (int)nb;
        }
        if (!barrier()) return;
        for (int64_t e = tid; e < nb; e += nt) A.bsorted[atomicAdd(&A.bcnt[A.bcell[e]], 1)] = A.blist[e];
        if (!barrier()) return;
        const int64_t occ = *(volatile unsigned*)&C->occ[bp];
        const bool dense = nb >= 2 * occ, wide = nb >= 16 * occ;
        // squared diagonal of a cell below every v of the band (grid coordinates are the points' own up to 3-D)
        const bool within = A.d <= 3 && gb.c * gb.c * gb.dg * (1.0 + 1e-9) < T;
        for (;; ++round) {
            const int rp = round % 3;
            // whether the block saw an active point: one store per block (a store per point
            // to the one word took 0.1 ms a round at 2^20 points)
            if (threadIdx.x == 0) active = 0;
            __syncthreads();
            auto post_active = [&]() {
                __syncthreads();
                if (threadIdx.x == 0 && active) C->nact[rp] = 1u;
            };
            // per band cell the largest value (as bits) of its undecided points, -1 if none: a
            // dominance scan skips the cells whose largest value is below its own
            // Dense bands (several points an occupied cell): 8 or 32 lanes per cell find its
            // undecided point of largest key.  That point dominates the others of its
            // cell, surely so where the cell's diagonal is below every sqrt(v) of the
            // band, else if the distance says so; only what is left is looked at by a
            // warp below.  (A thread per band point spent most of a round on points near
            // the top of their cells.)
            if (dense) {
                const int lg = wide ? 32 : 8, l8 = lane & (lg - 1), per_warp = 32 / lg;
                for (int64_t c4 = warp * per_warp; c4 < gb.ncells; c4 += nw * per_warp) {
                    const int64_t c = c4 + lane / lg;
                    const int f0 = c < gb.ncells ? A.bstart[c] : 0, f1 = c < gb.ncells ? A.bstart[c + 1] : 0;
                    Cand best{0.0, 0, -1};
                    for (int f = f0 + l8; f < f1; f += lg) {
                        const int p = A.bsorted[f];
                        if (A.stat[p] == 0) best.take(A.v2[p], A.idg[p], p);
                    }
                    __syncwarp();
                    if (wide && lane == 0) beat(A);
                    if (wide) best.warp_best();
                    else best.best_of<4>();
                    const bool act = best.g >= 0 && best.v >= T;
                    if (l8 == 0 && c < gb.ncells) {
                        A.cmax[c] = best.g >= 0 ? vbits(best.v) : -1;
                        A.champ[c] = act ? best.g : -1;
                        if (act) active = 1;
                    }
                    if (!within && act)
                        for (int f = f0 + l8; f < f1; f += lg) {
                            const int p = A.bsorted[f];
                            if (p == best.g || A.stat[p] != 0) continue;
                            const double vp = A.v2[p];
                            if (!(vp >= T)) continue;
                            const int sc = screen_rows<HIGH>(A.xgf + (int64_t)p * A.df, A.xgf + (int64_t)best.g * A.df, A.d,
                                                      sqrtf((float)vp), A.delta);
                            if (sc > 0) continue;
                            if (sc == 0 || !(dist2_exact(A.xg + (int64_t)p * A.d, A.xg + (int64_t)best.g * A.d, A.d) < vp))
                                A.hard[list_slot(&C->nhard[rp])] = p;
                        }
                    __syncwarp();
                }
                post_active();
                if (!barrier()) return;
            }
            // Otherwise: per band cell the largest value (as bits) of its undecided points,
            // -1 if none (a scan skips the cells whose largest value is below its own), ...
            if (!dense) {
                for (int64_t c = tid; c < gb.ncells; c += nt) {
                    long long m = -1;
                    for (int f = A.bstart[c]; f < A.bstart[c + 1]; ++f) {
                        if ((f & 4095) == 4095) beat(A);
                        const int p = A.bsorted[f];
                        if (A.stat[p] == 0) m = max(m, vbits(A.v2[p]));
                    }
                    A.cmax[c] = m;
                }
                if (!barrier()) return;
            }
            // ... then a thread per band point; the long scans are handed to a warp each
            for (int64_t e = dense ? nb : tid; e < nb; e += nt) {
                const int q = A.bsorted[e];
                if (A.stat[q] != 0) continue;
                const double vq = A.v2[q];
                if (!(vq >= T)) continue;
                active = 1;
                beat(A);
                // the point that dominated it before may still do
                const int w0 = A.wit[q];
                if (w0 >= 0 && A.stat[w0] == 0 && A.wd[q] < vq && key_above(A.v2[w0], A.idg[w0], vq, A.idg[q])) continue;
                double wd = 0.0;
                const int k = dominator_thread<HIGH>(A, gb, q, vq, DOM_THREAD_BUDGET, wd);
                if (k == -1) A.sel[list_slot(&C->nsel[rp])] = q;
                else if (k == -2) A.hard[list_slot(&C->nhard[rp])] = q;
                else {
                    A.wit[q] = k;
                    A.wd[q] = wd;
                }
            }
            if (!dense) {
                post_active();
                if (!barrier()) return;
            }
            if (*(volatile unsigned*)&C->nact[rp] == 0u) break;  // band exhausted
            int64_t nh = *(volatile unsigned*)&C->nhard[rp];
            const int32_t* left = A.hard;
            if (HIGH && dense && nh > nw) {
                // More points left than warps: a thread each looks at the nearest few
                // candidates first.  Where points spread over many dimensions, their cells
                // hold points that are far apart, so few are dominated by their cell's
                // largest one, but most by one of the next few; a warp a point spent
                // 843 of the 990 ms of 60,000 points in the cube of R^20 on them.
                for (int64_t e = tid; e < nh; e += nt) {
                    const int q = A.hard[e];
                    beat(A);
                    const double vq = A.v2[q];
                    const int w0 = A.wit[q];
                    if (w0 >= 0 && A.stat[w0] == 0 && A.wd[q] < vq && key_above(A.v2[w0], A.idg[w0], vq, A.idg[q])) continue;
                    double wd = 0.0;
                    const int k = dominator_thread<HIGH>(A, gb, q, vq, LIST_BUDGET, wd);
                    if (k == -1) A.sel[list_slot(&C->nsel[rp])] = q;
                    else if (k == -2) A.blist[list_slot(&C->nlong[rp])] = q;
                    else {
                        A.wit[q] = k;
                        A.wd[q] = wd;
                    }
                }
                if (!barrier()) return;
                nh = *(volatile unsigned*)&C->nlong[rp];
                left = A.blist;
            }
            auto scan = [&](int q) {
                if (lane == 0) beat(A);
                double wd = 0.0;
                const double vq = A.v2[q];
                const int k = dense ? dominator_warp<HIGH, true>(A, gb, q, vq, wd) : dominator_warp<HIGH, false>(A, gb, q, vq, wd);
                if (lane == 0) {
                    if (k == -1) {
                        A.sel[atomicAdd(&C->nsel[rp], 1u)] = q;
                    } else {
                        A.wit[q] = k;
                        A.wd[q] = wd;
                    }
                }
            };
            if (dense)  // the cells' largest points: cells warp, warp + nw, ..., 32 looked up at a time
                for (int64_t cb = warp; cb < gb.ncells; cb += 32 * nw) {
                    const int64_t c = cb + lane * nw;
                    const int mine = c < gb.ncells ? A.champ[c] : -1;
                    for (unsigned m = __ballot_sync(0xffffffffu, mine >= 0); m; m &= m - 1)
                        scan(__shfl_sync(0xffffffffu, mine, __ffs(m) - 1));
                }
            for (int64_t e = warp; e < nh; e += nw) scan(left[e]);
            if (!barrier()) return;
            // lower v2 of the undecided points of smaller key around every selected point: W
            // warps a point.  A point selected in this
            // round has no larger undecided key within its reach, so it does not matter
            // whether it is marked yet.
            const int64_t ns = *(volatile unsigned*)&C->nsel[rp];
            if (ns == 0) {
                if (first) atomicCAS(&C->status, 0, DEV_BAD_INPUT);
                return;
            }
            if (first) {
                const int nx = (round + 1) % 3;
                C->nsel[nx] = C->nact[nx] = C->nhard[nx] = C->nlong[nx] = 0u;
                C->rounds = round + 1;
            }
            constexpr int UPD = 2;
            const int64_t W = max((int64_t)1, min((int64_t)64, nw / ns));
            for (int64_t u = warp; u < ns * W; u += nw) {
                const int p = A.sel[u / W];
                const int part = (int)(u % W);
                if (part == 0 && lane == 0) A.stat[p] = 1;
                const double* xp = A.xg + (int64_t)p * A.d;
                const double vp = A.v2[p];  // final value of the selected point
                const int idp = A.idg[p];
                const int4 pc = A.pcell[p];
                const int sx = span_of_v(A.g0, vp, inv_c0, 0);
                const int x0 = max(0, pc.x - sx), x1 = min(A.g0.n[0] - 1, pc.x + sx);
                int y0 = 0, y1 = 0, z0 = 0, z1 = 0;
                if (A.g0.dg > 1) {
                    const int sy = span_of_v(A.g0, vp, inv_c0, 1);
                    y0 = max(0, pc.y - sy);
                    y1 = min(A.g0.n[1] - 1, pc.y + sy);
                }
                if (A.g0.dg > 2) {
                    const int sz = span_of_v(A.g0, vp, inv_c0, 2);
                    z0 = max(0, pc.z - sz);
                    z1 = min(A.g0.n[2] - 1, pc.z + sz);
                }
                // the rows of cells of the box in batches of rb: a lane per row finds where its
                // points start, and the batch's points go to the lanes in one sequence
                const int ny = y1 - y0 + 1, rows = ny * (z1 - z0 + 1);
                const int rb = max(1, min(32, (rows + (int)W - 1) / (int)W));
                for (int r0 = part * rb; r0 < rows; r0 += (int)W * rb) {
                    if (lane == 0) beat(A);
                    const int r = r0 + lane;
                    int64_t a = 0;
                    int len = 0;
                    if (lane < rb && r < rows) {
                        const int64_t base = ((int64_t)(z0 + r / ny) * A.g0.n[1] + y0 + r % ny) * A.g0.n[0];
                        a = A.cstart[base + x0];
                        len = (int)(A.cstart[base + x1 + 1] - a);
                    }
                    int inc = len;
#pragma unroll
                    for (int o = 1; o < 32; o <<= 1) {
                        const int up = __shfl_up_sync(0xffffffffu, inc, o);
                        if (lane >= o) inc += up;
                    }
                    const int total = __shfl_sync(0xffffffffu, inc, 31);
                    // UPD points a lane, places at[] (-1: none), so that their loads overlap (one at a
                    // time: 1238 against 1152 ms for 100,000 points with heavy tails, whose grid has
                    // most points in a few cells)
                    auto lower = [&](const int64_t (&at)[UPD]) {
                        int st[UPD];
                        double v[UPD];
#pragma unroll
                        for (int u = 0; u < UPD; ++u) {
                            st[u] = at[u] >= 0 ? A.stat[at[u]] : 1;
                            v[u] = at[u] >= 0 ? A.v2[at[u]] : 0.0;
                        }
#pragma unroll
                        for (int u = 0; u < UPD; ++u) {
                            const int64_t q = at[u];
                            const double vq = v[u];
                            if (st[u] != 0 || !(vq < vp || (vq == vp && A.idg[q] > idp))) continue;
                            if (screen_rows<HIGH>(A.xgf + q * A.df, A.xgf + (int64_t)p * A.df, A.d, sqrtf((float)vq), A.delta) == 0)
                                continue;
                            const double dd = dist2_exact(A.xg + q * A.d, xp, A.d);
                            if (dd < vq)
                                atomicMin((unsigned long long*)A.v2 + q, (unsigned long long)__double_as_longlong(dd));
                        }
                    };
                    if (HIGH && total >= 32 * min(rb, rows - r0)) {  // long rows one by one, without the search
                        for (int k = 0; k < min(rb, rows - r0); ++k) {
                            const int64_t ra = __shfl_sync(0xffffffffu, a, k);
                            const int ln = __shfl_sync(0xffffffffu, len, k);
                            for (int m = lane; m < ln; m += 32 * UPD) {
                                if (lane == 0 && (m & 2047) == 2048 - 32 * UPD) beat(A);
                                int64_t at[UPD];
#pragma unroll
                                for (int u = 0; u < UPD; ++u) at[u] = m + 32 * u < ln ? ra + m + 32 * u : -1;
                                lower(at);
                            }
                        }
                        continue;
                    }
                    for (int m0 = 0; m0 < total; m0 += 32 * UPD) {
                        if (lane == 0 && (m0 & 2047) == 2048 - 32 * UPD) beat(A);
                        int64_t at[UPD];
#pragma unroll
                        for (int u = 0; u < UPD; ++u) {
                            const int m = m0 + 32 * u + lane;
                            const int row = which_row(inc, m);
                            const int64_t ra = __shfl_sync(0xffffffffu, a, row);
                            const int rs = __shfl_sync(0xffffffffu, inc - len, row);
                            at[u] = m < total ? ra + (m - rs) : -1;
                        }
                        lower(at);
                    }
                }
            }
            if (!barrier()) return;
        }
        ++round;  // its counters are used: selected none, so they stay as they are
        if (first) {
            const int nx = round % 3;
            C->nsel[nx] = C->nact[nx] = C->nhard[nx] = C->nlong[nx] = 0u;
        }
    }
}

__global__ void ord_cells_k(Grid g, const double* __restrict__ gxg, int gs, int64_t N, int4* __restrict__ pcell) {
    const int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= N) return;
    int c[3] = {0, 0, 0};
    for (int t = 0; t < g.dg; ++t) c[t] = cell_coord(g, gxg[q * gs + t], t);
    pcell[q] = make_int4(c[0], c[1], c[2], 0);
}

__global__ void ord_keys_k(const double* __restrict__ v2, const int32_t* __restrict__ idg, int64_t N,
                           uint64_t* __restrict__ key, int64_t* __restrict__ val) {
    int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= N) return;
    int64_t id = idg[q];
    key[id] = ~(uint64_t)__double_as_longlong(v2[q]);
    val[id] = id;
}

__global__ void ord_out_k(const uint64_t* __restrict__ skey, const int64_t* __restrict__ sval, const double* __restrict__ x,
                          int64_t N, int d, int32_t* __restrict__ perm, double* __restrict__ l,
                          double* __restrict__ x_ord) {
    int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= N) return;
    int64_t id = sval[k];
    perm[k] = (int32_t)id;
    double v = __longlong_as_double((long long)~skey[k]);
    l[k] = __dsqrt_rn(v);
    for (int t = 0; t < d; ++t) x_ord[k * d + t] = x[id * d + t];
}

// limit: cycles without a sign of work after which a wait of the kernels gives up.
kc_status order_impl(const double* x, int64_t N, int d, int32_t* perm, double* l, double* x_ord, long long limit,
                     cudaStream_t s) {
    Arena A(s);
    Origin org, top;
    double E = 0.0;
    KC_TRY(points_bounds(x, N, d, &org, &top, &E, A, s));
    // grid coordinates: the points (d <= 3) or their principal-axes projections
    const double* gx;
    int gs;
    double beyond = 0.0;  // share of the points' variance outside the grid's axes
    KC_TRY(grid_coords(x, N, d, A, s, &gx, &gs, &beyond));
    double lo[3] = {org.lo[0], org.lo[1], org.lo[2]}, hi[3] = {top.lo[0], top.lo[1], top.lo[2]};
    if (gx != x) KC_TRY(bbox(gx, N, gs, lo, hi, A, s));
    // fine grid of all points, about two points per cell
    Grid g0 = make_grid(gs, lo, hi, N, 0.0, N / 2 > 1 ? N / 2 : 1);
    int32_t* gsorted;
    int64_t* cstart;
    KC_TRY(A.get(&gsorted, N));
    KC_TRY(A.get(&cstart, g0.ncells + 1));
    KC_TRY(grid_build(g0, gx, gs, nullptr, N, gsorted, cstart, A, s));

    double *xg, *v2;
    int32_t* idg;
    int* stat;
    KC_TRY(A.get(&xg, N * d));
    KC_TRY(A.get(&v2, N));
    KC_TRY(A.get(&idg, N));
    KC_TRY(A.get(&stat, N));
    // float copy of the coordinates (minus the box corner) for FP32 screens of
    // the distance tests; exact FP64 tests decide every close call
    float* xgf = nullptr;
    // 2^-23 E; infinite, so that only exact tests decide, where floats could over- or underflow
    const float delta = E > 1e-12 && E < 1e18 ? (float)(E * 1.1920928955078125e-07) : INFINITY;
    KC_TRY(A.get(&xgf, N * row_floats(d)));
    ::kc::note_launch(), ord_init_k<<<blocks_for(N, 256), 256, 0, s>>>(x, d, gsorted, N, xg, idg, v2, stat, org, xgf);
    // grid coordinates in grid order
    const double* gxg = xg;
    if (gx != x) {
        double* p;
        KC_TRY(A.get(&p, (size_t)N * gs));
        ::kc::note_launch(), gather_rows_k<<<blocks_for(N, 256), 256, 0, s>>>(gx, gs, gsorted, N, p);
        gxg = p;
    }
    int4* pcell;
    KC_TRY(A.get(&pcell, N));
    ::kc::note_launch(), ord_cells_k<<<blocks_for(N, 256), 256, 0, s>>>(g0, gxg, gs, N, pcell);
    KC_CUDA(cudaGetLastError());
    const int sms = sm_count();

    // Greedy phase: the coarsest points are selected one at a time (every
    // step updates every point), because while few points are selected the
    // update balls cover the whole cloud and the band rounds would be
    // quadratic.
    BandCtl* ctl;
    KC_TRY(A.get(&ctl, 1));
    KC_CUDA(cudaMemsetAsync(ctl, 0, sizeof(BandCtl), s));
    {
        // one block, which exchanges nothing, for up to 4 points a thread
        const int nblk = N <= 4 * GREEDY_THREADS ? 1 : (int)std::min<int64_t>(sms, (N + GREEDY_THREADS - 1) / GREEDY_THREADS);
        ulonglong2* slots;
        KC_TRY(A.get(&slots, 2 * nblk * nblk));
        KC_CUDA(cudaMemsetAsync(slots, 0, sizeof(ulonglong2) * 2 * nblk * nblk, s));
        const int64_t most = beyond > 0.05 ? GREEDY_STEPS_SPREAD : GREEDY_STEPS;
        int64_t steps = N - 1 < most ? N - 1 : most;
        const double* a_xg = xg;
        const int32_t* a_idg = idg;
        const float* a_xgf = xgf;
        int* gst = &ctl->status;
        long long lim = limit;
        float dl = delta;
        void* args[] = {(void*)&a_xg, (void*)&d, (void*)&a_idg, (void*)&v2, (void*)&stat, (void*)&N, (void*)&steps,
                        (void*)&slots, (void*)&a_xgf, (void*)&dl, (void*)&gst, (void*)&lim};
        auto gfn = d > 3 ? ord_greedy_loop_k<true> : ord_greedy_loop_k<false>;
        ::kc::note_launch();
        KC_CUDA(cudaLaunchCooperativeKernel((const void*)gfn, dim3(nblk), dim3(GREEDY_THREADS), args, 0, s));
    }
    {
        BandArgs a;
        a.N = N;
        a.d = d;
        a.df = row_floats(d);
        a.gs = gs;
        a.g0 = g0;
        a.cstart = cstart;
        a.xg = xg;
        a.xgf = xgf;
        a.gxg = gxg;
        a.pcell = pcell;
        a.idg = idg;
        a.delta = delta;
        a.v2 = v2;
        a.stat = stat;
        a.ctl = ctl;
        a.limit = limit;
        a.beat_shift = 0;
        while ((32LL << a.beat_shift) <= limit) ++a.beat_shift;
        for (int t = 0; t < 3; ++t) {
            a.lo[t] = t < g0.dg ? lo[t] : 0.0;
            a.hi[t] = t < g0.dg ? hi[t] : 0.0;
        }
        KC_TRY(A.get(&a.blist, N));
        KC_TRY(A.get(&a.bcell, N));
        KC_TRY(A.get(&a.bsorted, N));
        KC_TRY(A.get(&a.hard, N));
        KC_TRY(A.get(&a.sel, N));
        KC_TRY(A.get(&a.bcnt, 2 * N + 1));    // a band of nb points has at most 2 nb + 1 cells
        KC_TRY(A.get(&a.bstart, 2 * N + 2));
        KC_TRY(A.get(&a.cmax, 2 * N + 1));
        KC_TRY(A.get(&a.champ, 2 * N + 1));
        KC_TRY(A.get(&a.wit, N));
        KC_TRY(A.get(&a.wd, N));
        KC_CUDA(cudaMemsetAsync(a.wit, 0xff, sizeof(int32_t) * N, s));  // -1
        auto kfn = d > 3 ? ord_bands_k<true> : ord_bands_k<false>;
        int per_sm = 0;
        KC_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kfn, 256, 0));
        // A block per 256 points (few blocks keep the barriers short), at most what is resident
        // at once.  Past three dimensions a block per 16: a round's scans take longer than its
        // barriers there (5000 points in R^20: 32.3 ms with a block per 256, 20.7 with one per
        // 64 or 16; 10,000 of a swiss roll 5.5, 4.8 and 3.1).
        const int nblk = (int)std::min<int64_t>((int64_t)sms * std::max(1, per_sm), d > 3 ? (N + 15) / 16 : (N + 255) / 256);
        KC_TRY(A.get(&a.part, nblk));
        KC_TRY(A.get(&a.flags, nblk * BAR_STRIDE));
        KC_CUDA(cudaMemsetAsync(a.flags, 0, sizeof(unsigned) * nblk * BAR_STRIDE, s));
        void* args[] = {(void*)&a};
        ::kc::note_launch();
        KC_CUDA(cudaLaunchCooperativeKernel((const void*)kfn, dim3(nblk), dim3(256), args, 0, s));
        BandCtl h;
        KC_CUDA(cudaMemcpyAsync(&h, ctl, sizeof(h), cudaMemcpyDeviceToHost, s));
        KC_CUDA(cudaStreamSynchronize(s));
        if (h.status == DEV_TIMEOUT) return fail(KC_ETIMEOUT, "ordering: a grid barrier ran out");
        if (h.status != 0) return fail(KC_ECUDA, "ordering: no dominant point in a nonempty band");
        if (getenv("KC_ORDER_STATS")) fprintf(stderr, "[kc order] N=%lld rounds=%d\n", (long long)N, h.rounds);
    }
    uint64_t *k0, *k1;
    int64_t *w0, *w1;
    KC_TRY(A.get(&k0, N));
    KC_TRY(A.get(&k1, N));
    KC_TRY(A.get(&w0, N));
    KC_TRY(A.get(&w1, N));
    ::kc::note_launch(), ord_keys_k<<<blocks_for(N, 256), 256, 0, s>>>(v2, idg, N, k0, w0);
    KC_TRY(radix_sort_u64_i64(k0, w0, k1, w1, N, 64, A, s));
    ::kc::note_launch(), ord_out_k<<<blocks_for(N, 256), 256, 0, s>>>(k1, w1, x, N, d, perm, l, x_ord);
    KC_CUDA(cudaGetLastError());
    KC_CUDA(cudaStreamSynchronize(s));
    return KC_OK;
}

}  // namespace kc
