// a4: the dependency schedule of the factorisation.
//
// Column i of the left-looking ICHOL(0) (Algorithm 2) needs every column k in
// row i of L (k in R_i) to be complete, so the columns form a DAG whose
// levels are level(i) = 1 + max_{k in R_i} level(k).  This file builds, on the
// device: the CSC view of L (rows of each column ascending, with the CSR slot
// of every entry), the levels (a sync-free kernel over rows in index order),
// and the columns sorted by level with a stable radix sort; within a level by
// index, or, given the points, by the Morton code of each column's point, so
// that the factor's consecutive tasks and the solves' consecutive rows touch
// neighbouring points, whose rows share most of their entries (L2 reuse).
#include <algorithm>
#include <climits>

#include "grid.cuh"

namespace kc {

// ------------------------------------------------------------- CSC view
// The CSR entries in stable order of their columns: a radix sort by digits of
// the column index, written for this use.  An item is (column, (row, place in
// the row)); the first pass makes the items from the rows themselves, the last
// one writes rowidx, slot and colptr, so that 188.7 M entries (2^20 points,
// rho = 3; 20-bit columns, three passes) move 60 bytes an entry instead of 124
// with 64-bit items, a pass that lays them out and one that takes them apart: 4.2
// ms instead of 6.9.  Bound by the ranking and the turn through shared memory
// (1.1 to 1.5 ms a scatter for 3 to 4.5 GB) at 32 warps an SM: 24 warps without
// spills take 0.3 ms more over the three passes, two passes by 10-bit digits 2 ms.
//
// A tile is 8 warps x 16 rounds x 32 lanes, every warp owning 512 consecutive
// entries processed in order; histograms are digit-major, hist[digit][tile].
constexpr int CS_WARPS = 8, CS_ROUNDS = 16, CS_RUN = CS_ROUNDS * 32, CS_TILE = CS_WARPS * CS_RUN;
constexpr int CS_DIGIT = 8, CS_ND = 1 << CS_DIGIT;  // digits of at most CS_DIGIT bits
constexpr int CS_PER = CS_ND / (CS_WARPS * 32);                // digits per thread

// runrow[t] = the row of entry t * CS_RUN; the longest row; colptr ready for the
// last pass's minima
__global__ void csc_rows_k(const int64_t* __restrict__ rowptr, int64_t N, int64_t nnz, int32_t* __restrict__ runrow,
                           int* __restrict__ longest, long long* __restrict__ colptr) {
    const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    int len = 0;
    if (j < N) {
        const int64_t a = rowptr[j], b = rowptr[j + 1];
        len = (int)(b - a);
        colptr[j] = LLONG_MAX;
        if (j == 0) colptr[N] = nnz;
        for (int64_t t = (a + CS_RUN - 1) / CS_RUN; t * CS_RUN < b; ++t) runrow[t] = (int32_t)j;
    }
    len = __reduce_max_sync(0xffffffffu, len);
    if (lane_id() == 0 && len > 0) atomicMax(longest, len);
}

__global__ void __launch_bounds__(CS_WARPS * 32) csc_hist_k(const uint32_t* __restrict__ key, int64_t n, int shift,
                                                            int nd, int64_t ntiles, int32_t* __restrict__ hist) {
    __shared__ int cnt[CS_ND];
    for (int i = threadIdx.x; i < nd; i += blockDim.x) cnt[i] = 0;
    __syncthreads();
    const int64_t base = (int64_t)blockIdx.x * CS_TILE;
    const int m = (int)min((int64_t)CS_TILE, n - base);
#pragma unroll 4
    for (int i = threadIdx.x; i < m; i += CS_WARPS * 32) atomicAdd(&cnt[(key[base + i] >> shift) & (nd - 1)], 1);
    __syncthreads();
    for (int i = threadIdx.x; i < nd; i += blockDim.x) hist[(int64_t)i * ntiles + blockIdx.x] = cnt[i];
}

struct CscArgs {
    const int64_t* rowptr;
    const uint32_t* kin;    // keys (the first pass: the CSR columns)
    const void* vin;        // items (not read by the first pass)
    const int32_t* runrow;  // (first pass)
    int64_t N, nnz, ntiles;
    const int64_t* goff;    // scanned histograms
    uint32_t* kout;
    void* vout;
    long long* colptr;      // (last pass)
    int32_t* rowidx;
    int64_t* slot;
    int shift, nd;
    int pb;                 // bits of an item's place in its row
};

// Ranks its tile's entries by digit (match_any, in entry order: stable), turns
// the tile into digit order in shared memory and writes every digit's run to its
// place, consecutive threads to consecutive addresses.
template <typename V, bool FIRST, bool LAST>
__global__ void __launch_bounds__(CS_WARPS * 32, sizeof(V) == 4 ? 4 : 3) csc_scatter_k(CscArgs A) {
    extern __shared__ __align__(16) unsigned char cs_smem[];
    V* sval = (V*)cs_smem;                         // [CS_TILE]
    uint32_t* skey = (uint32_t*)(sval + CS_TILE);  // [CS_TILE]
    __shared__ int wcnt[CS_WARPS][CS_ND];          // per-warp digit counts, then the warps' starts in the tile
    __shared__ int dstart[CS_ND];                  // tile-local start of every digit
    __shared__ long long gbase[CS_ND];             // global start of every digit of this tile
    __shared__ int wsum[CS_WARPS];
    const unsigned FULL = 0xffffffffu;
    const int lane = lane_id(), w = threadIdx.x >> 5;
    for (int i = lane; i < A.nd; i += 32) wcnt[w][i] = 0;
    __syncwarp();
    const int64_t tbase = (int64_t)blockIdx.x * CS_TILE;
    const int cnt = (int)min((int64_t)CS_TILE, A.nnz - tbase), w0 = w * CS_RUN;  // places in the tile below
    const unsigned lt = (1u << lane) - 1u;
    uint32_t kr[CS_ROUNDS];
    unsigned rank[CS_ROUNDS / 2];  // places among the warp's entries of the same digit, two a word
    [[maybe_unused]] V vr[FIRST ? CS_ROUNDS : 1];
#pragma unroll
    for (int r = 0; r < CS_ROUNDS; ++r) {
        const int i = w0 + r * 32 + lane;
        kr[r] = i < cnt ? A.kin[tbase + i] : 0u;
    }
    if constexpr (FIRST) {
        // the entries' rows: row = the row of the round's first entry, then one more at
        // every row start among the 32 entries; a round with an empty row in it (a row
        // that lacks its diagonal) looks every entry's row up
        if (w0 < cnt) {
            int row = A.runrow[(tbase + w0) / CS_RUN];
            int64_t start = A.rowptr[row];
            const int nrows = (int)A.N;
#pragma unroll
            for (int r = 0; r < CS_ROUNDS; ++r) {
                const int64_t e0 = tbase + w0 + r * 32;
                const int next = row + 1 + lane;
                const int64_t nb = A.rowptr[min(nrows, next)];
                const int off = next < nrows ? (int)max((int64_t)0, min(nb - e0, (int64_t)64)) : 64;
                const unsigned bits = __reduce_or_sync(FULL, off > 0 && off < 32 ? 1u << off : 0u);
                if (__popc(__ballot_sync(FULL, off < 32)) != __popc(bits)) {
                    int64_t a = 0, b = nrows - 1;  // the last row that starts at or before the entry
                    while (a < b) {
                        const int64_t mid = (a + b + 1) >> 1;
                        if (A.rowptr[mid] <= e0 + lane) a = mid;
                        else b = mid - 1;
                    }
                    vr[r] = ((V)a << A.pb) | ((V)(e0 + lane - A.rowptr[a]) & (((V)1 << A.pb) - 1));
                    row = __shfl_sync(FULL, (int)a, 31);
                    start = A.rowptr[row];
                    continue;
                }
                const unsigned mine = bits & (lt | (1u << lane));
                const unsigned pos = mine ? (unsigned)(lane - (31 - __clz(mine))) : (unsigned)(e0 + lane - start);
                vr[r] = ((V)(row + __popc(mine)) << A.pb) | (V)pos;
                // the next round's row: the last row start at or before e0 + 32
                const int np = __popc(__ballot_sync(FULL, off <= 32));
                if (np) {
                    start = __shfl_sync(FULL, nb, np - 1);
                    row += np;
                }
            }
        }
    }
#pragma unroll
    for (int r = 0; r < CS_ROUNDS; ++r) {
        const bool ok = w0 + r * 32 + lane < cnt;
        const int dg = ok ? (int)((kr[r] >> A.shift) & (unsigned)(A.nd - 1)) : CS_ND + lane;
        const unsigned peers = __match_any_sync(FULL, dg);
        const int before = ok ? wcnt[w][dg] : 0;
        __syncwarp();
        if (ok && lane == 31 - __clz(peers)) wcnt[w][dg] = before + __popc(peers);
        const unsigned at = before + __popc(peers & lt);
        if (r & 1) rank[r / 2] |= at << 16;
        else rank[r / 2] = at;
        __syncwarp();
    }
    __syncthreads();
    // digit totals of the tile, their exclusive scan, and the per-warp offsets
    {
        const int d0 = threadIdx.x * CS_PER;
        int tot[CS_PER], sum = 0;
#pragma unroll
        for (int u = 0; u < CS_PER; ++u) {
            tot[u] = 0;
            if (d0 + u < A.nd)
                for (int q = 0; q < CS_WARPS; ++q) tot[u] += wcnt[q][d0 + u];
            sum += tot[u];
        }
        int incl = sum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(FULL, incl, o);
            if (lane >= o) incl += y;
        }
        if (lane == 31) wsum[w] = incl;
        __syncthreads();
        int run = incl - sum;
        for (int q = 0; q < w; ++q) run += wsum[q];
#pragma unroll
        for (int u = 0; u < CS_PER; ++u) {
            const int dg = d0 + u;
            if (dg < A.nd) {
                dstart[dg] = run;
                gbase[dg] = A.goff[(int64_t)dg * A.ntiles + blockIdx.x] - run;
                int at = run;
                for (int q = 0; q < CS_WARPS; ++q) {
                    const int c = wcnt[q][dg];
                    wcnt[q][dg] = at;
                    at += c;
                }
            }
            run += tot[u];
        }
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < CS_ROUNDS; ++r) {
        const int i = w0 + r * 32 + lane;
        if (i < cnt) {
            const int dg = (int)((kr[r] >> A.shift) & (unsigned)(A.nd - 1));
            const int at = wcnt[w][dg] + (int)((rank[r / 2] >> (r & 1 ? 16 : 0)) & 0xffffu);
            skey[at] = kr[r];
            if constexpr (FIRST) sval[at] = vr[r];
            else sval[at] = ((const V*)A.vin)[tbase + i];
        }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < cnt; i += CS_WARPS * 32) {
        const uint32_t k = skey[i];
        const V v = sval[i];
        const int dg = (int)((k >> A.shift) & (unsigned)(A.nd - 1));
        const long long q = gbase[dg] + i;
        if constexpr (LAST) {
            const int64_t row = (int64_t)(v >> A.pb);
            A.rowidx[q] = (int32_t)row;
            A.slot[q] = A.rowptr[row] + (int64_t)(v & (((V)1 << A.pb) - 1));
            // a digit's run ascends in the whole key: a column starts in this tile here
            if ((i == dstart[dg] || skey[i - 1] != k) && k < (unsigned)A.N) atomicMin(&A.colptr[k], q);
        } else {
            A.kout[q] = k;
            ((V*)A.vout)[q] = v;
        }
    }
}

static int bits_for(int64_t v) {
    int b = 1;
    while (b < 63 && ((int64_t)1 << b) <= v) ++b;
    return b;
}

template <typename V>
static kc_status csc_passes(CscArgs a, const int32_t* col, int pb, Arena& A, cudaStream_t s) {
    const int bits = bits_for(a.N - 1), passes = (bits + CS_DIGIT - 1) / CS_DIGIT;
    const int width = (bits + passes - 1) / passes;  // digits of even width: longer runs than 8, 8 and the rest
    uint32_t* k[2] = {nullptr, nullptr};
    V* v[2] = {nullptr, nullptr};
    int32_t* hist;
    int64_t* goff;
    KC_TRY(A.get(&hist, ((int64_t)1 << width) * a.ntiles));
    KC_TRY(A.get(&goff, ((int64_t)1 << width) * a.ntiles + 1));
    for (int t = 0; t < std::min(passes - 1, 2); ++t) {
        KC_TRY(A.get(&k[t], a.nnz));
        KC_TRY(A.get(&v[t], a.nnz));
    }
    const size_t smem = (size_t)CS_TILE * (sizeof(uint32_t) + sizeof(V));
    a.pb = pb;
    a.nd = 1 << width;
    a.goff = goff;
    for (int p = 0; p < passes; ++p) {
        a.shift = p * width;
        a.kin = p ? k[(p - 1) & 1] : (const uint32_t*)col;
        a.vin = p ? v[(p - 1) & 1] : nullptr;
        a.kout = k[p & 1];
        a.vout = v[p & 1];
        const bool last = p == passes - 1;
        auto kfn = p == 0 ? (last ? csc_scatter_k<V, true, true> : csc_scatter_k<V, true, false>)
                          : (last ? csc_scatter_k<V, false, true> : csc_scatter_k<V, false, false>);
        KC_TRY(allow_dynamic_smem(kfn));
        ::kc::note_launch(), csc_hist_k<<<(unsigned)a.ntiles, CS_WARPS * 32, 0, s>>>(a.kin, a.nnz, a.shift, a.nd,
                                                                                     a.ntiles, hist);
        KC_TRY(exclusive_scan_i32_to_i64(hist, goff, (int64_t)a.nd * a.ntiles, A, s));
        ::kc::note_launch(), kfn<<<(unsigned)a.ntiles, CS_WARPS * 32, smem, s>>>(a);
        KC_CUDA(cudaGetLastError());
    }
    return KC_OK;
}

static kc_status csc_view(int64_t N, const int64_t* rowptr, const int32_t* col, int64_t nnz, int64_t* colptr,
                          int32_t* rowidx, int64_t* slot, Arena& A, cudaStream_t s) {
    CscArgs a{};
    a.rowptr = rowptr;
    a.N = N;
    a.nnz = nnz;
    a.ntiles = (nnz + CS_TILE - 1) / CS_TILE;
    a.colptr = (long long*)colptr;
    a.rowidx = rowidx;
    a.slot = slot;
    int32_t* runrow;
    int* longest;
    KC_TRY(A.get(&runrow, (nnz + CS_RUN - 1) / CS_RUN));
    KC_TRY(A.get(&longest, 1));
    KC_CUDA(cudaMemsetAsync(longest, 0, sizeof(int), s));
    ::kc::note_launch(), csc_rows_k<<<blocks_for(N, 256), 256, 0, s>>>(rowptr, N, nnz, runrow, longest, a.colptr);
    KC_CUDA(cudaGetLastError());
    a.runrow = runrow;
    // Items of 32 bits where a row and a place in it fit (N = 2^20: rows of up to 4096
    // entries), of 64 bits otherwise: 4.2 against 4.9 ms for the 188.7 M entries.
    // Up to 65,536 rows any place fits; beyond, the longest row decides.
    const int rb = bits_for(N - 1);
    bool fits = 2 * rb <= 32;
    if (!fits && rb < 32) {
        int h = 0;
        KC_CUDA(cudaMemcpyAsync(&h, longest, sizeof(int), cudaMemcpyDeviceToHost, s));
        KC_CUDA(cudaStreamSynchronize(s));
        fits = rb + bits_for(h - 1) <= 32;
    }
    if (fits) return csc_passes<uint32_t>(a, col, 32 - rb, A, s);
    return csc_passes<uint64_t>(a, col, 32, A, s);
}

// level[j] = 1 + max level over row j; rows claimed in index order, so a row
// waits only on rows with smaller index that were claimed before it.
__device__ __forceinline__ int ld_relaxed_level(const int* p) {
    int v;
    asm volatile("ld.relaxed.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
// level[j] = 1 + max level over row j; rows claimed in index order, so a row
// waits only on rows with smaller index that were claimed before it.  Each
// lane reads up to 8 of the row's levels with relaxed loads all in flight
// together and spins (bounded, with back-off) only on those not yet set.
// Only the level values are read, so no acquire ordering is needed.
__global__ void levels_k(const int64_t* __restrict__ rowptr, const int32_t* __restrict__ col, int64_t N,
                         int* __restrict__ level, unsigned long long* __restrict__ ticket, int* __restrict__ depth,
                         int* __restrict__ status, long long spin_limit) {
    constexpr int D = 8;
    int lane = lane_id();
    for (;;) {
        unsigned long long t = 0;
        if (lane == 0) t = atomicAdd(ticket, 1ULL);
        t = __shfl_sync(0xffffffffu, t, 0);
        if ((int64_t)t >= N) return;
        if (ld_volatile_s32(status) != 0) return;
        const int64_t j = (int64_t)t;
        const int64_t a = rowptr[j];
        const int n = (int)(rowptr[j + 1] - 1 - a);
        int m = 0;
        bool ok = true;
        for (int e0 = 0; e0 < n; e0 += 32 * D) {
            int kk[D], v[D];
#pragma unroll
            for (int u = 0; u < D; ++u) {
                const int e = e0 + lane + 32 * u;
                kk[u] = e < n ? __ldg(&col[a + e]) : -1;
            }
#pragma unroll
            for (int u = 0; u < D; ++u) v[u] = kk[u] >= 0 ? ld_relaxed_level(&level[kk[u]]) : 0;
#pragma unroll
            for (int u = 0; u < D; ++u) {
                if (kk[u] >= 0 && v[u] == 0 && ok) {
                    const long long t0 = clock64();
                    unsigned ns = 32;
                    while ((v[u] = ld_relaxed_level(&level[kk[u]])) == 0) {
                        if (clock64() - t0 > spin_limit || ld_volatile_s32(status) != 0) {
                            ok = false;
                            break;
                        }
                        __nanosleep(ns);
                        if (ns < 512) ns <<= 1;
                    }
                }
                m = max(m, v[u]);
            }
            if (!__all_sync(0xffffffffu, ok)) break;
        }
        if (!__all_sync(0xffffffffu, ok)) {
            if (lane == 0) atomicCAS(status, 0, DEV_TIMEOUT);
            return;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
        if (lane == 0) {
            st_release_s32(&level[j], m + 1);
            atomicMax(depth, m + 1);
        }
    }
}
__global__ void level_keys_k(const int* __restrict__ level, int64_t N, uint32_t* __restrict__ key,
                             int64_t* __restrict__ val) {
    int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (j < N) {
        key[j] = (uint32_t)level[j];
        val[j] = j;
    }
}

__global__ void level_morton_keys_k(const int* __restrict__ level, const double* __restrict__ x, int d, Box3 box,
                                    int64_t N, uint64_t* __restrict__ key, int64_t* __restrict__ val) {
    int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (j < N) {
        key[j] = ((uint64_t)(uint32_t)level[j] << 32) | morton_of(x + j * d, d, box);
        val[j] = j;
    }
}
__global__ void order_out_k(const int64_t* __restrict__ sval, int64_t N, int32_t* __restrict__ order) {
    int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p < N) order[p] = (int32_t)sval[p];
}

#ifndef KC_LEVELS_BLOCKS_PER_SM
#define KC_LEVELS_BLOCKS_PER_SM 2
#endif

// A second stream for work that runs beside the caller's stream `home`:
// fork() makes it wait for the work enqueued on home so far, join() makes
// home wait for it.  Going out of scope joins (if not joined yet) and
// releases the stream and events, so that scratch freed on home afterwards
// (an Arena declared before this object) is never freed under the second
// stream's work, whichever way the function returns.
struct AuxStream {
    cudaStream_t home = nullptr, s = nullptr;
    cudaEvent_t ev[2] = {nullptr, nullptr};
    bool joined = true;
    kc_status fork(cudaStream_t from) {
        home = from;
        KC_CUDA(cudaEventCreateWithFlags(&ev[0], cudaEventDisableTiming));
        KC_CUDA(cudaEventCreateWithFlags(&ev[1], cudaEventDisableTiming));
        KC_CUDA(cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking));
        KC_CUDA(cudaEventRecord(ev[0], from));
        KC_CUDA(cudaStreamWaitEvent(s, ev[0], 0));
        joined = false;
        return KC_OK;
    }
    kc_status join() {
        if (joined) return KC_OK;
        joined = true;
        KC_CUDA(cudaEventRecord(ev[1], s));
        KC_CUDA(cudaStreamWaitEvent(home, ev[1], 0));
        return KC_OK;
    }
    ~AuxStream() {
        if (!joined && s) {
            cudaEventRecord(ev[1], s);
            cudaStreamWaitEvent(home, ev[1], 0);
        }
        for (cudaEvent_t e : ev)
            if (e) cudaEventDestroy(e);
        if (s) cudaStreamDestroy(s);
    }
};

kc_status schedule_impl(int64_t N, const int64_t* rowptr, const int32_t* col, int64_t nnz, const double* x, int d,
                        int64_t* colptr, int32_t* rowidx, int64_t* slot, int32_t* level, int32_t* order,
                        int32_t* depth_out, cudaStream_t s) {
    Arena A(s);
    // The levels (a dependency chain, latency-bound) run on a second stream next to the CSC sort
    // (bound by its ranking): both read only the CSR rows.  The level kernel takes a quarter of the
    // SMs' thread slots so that the sort's blocks find room.
    unsigned long long* ticket;
    int* dev_depth;
    int* status;
    KC_TRY(A.get(&ticket, 1));
    KC_TRY(A.get(&dev_depth, 1));
    KC_TRY(A.get(&status, 1));
    KC_CUDA(cudaMemsetAsync(ticket, 0, sizeof(unsigned long long), s));
    KC_CUDA(cudaMemsetAsync(dev_depth, 0, sizeof(int), s));
    KC_CUDA(cudaMemsetAsync(status, 0, sizeof(int), s));
    KC_CUDA(cudaMemsetAsync(level, 0, sizeof(int) * N, s));
    AuxStream aux;
    KC_TRY(aux.fork(s));
    const int sms = sm_count();
    ::kc::note_launch(), levels_k<<<sms * KC_LEVELS_BLOCKS_PER_SM, 256, 0, aux.s>>>(rowptr, col, N, level, ticket,
                                                                               dev_depth, status, 4000000000LL);
    KC_CUDA(cudaGetLastError());

    KC_TRY(csc_view(N, rowptr, col, nnz, colptr, rowidx, slot, A, s));

    KC_TRY(aux.join());  // the levels are complete on s from here on
    int h_depth = 0, h_status = 0;
    KC_CUDA(cudaMemcpyAsync(&h_depth, dev_depth, sizeof(int), cudaMemcpyDeviceToHost, s));
    KC_CUDA(cudaMemcpyAsync(&h_status, status, sizeof(int), cudaMemcpyDeviceToHost, s));
    KC_CUDA(cudaStreamSynchronize(s));
    if (h_status != 0) return fail(KC_ETIMEOUT, "level computation: a dependency wait ran out");

    int64_t *v0, *v1;
    KC_TRY(A.get(&v0, N));
    KC_TRY(A.get(&v1, N));
    if (x) {
        // columns sorted by (level, Morton code of the point)
        double lo[3], hi[3];
        KC_TRY(bbox(x, N, d, lo, hi, A, s));
        Box3 box;
        for (int t = 0; t < 3; ++t) {
            box.lo[t] = t < d ? lo[t] : 0.0;
            const double e = t < d ? hi[t] - lo[t] : 0.0;
            box.inv[t] = e > 0 ? 1.0 / e : 0.0;
        }
        uint64_t *m0, *m1;
        KC_TRY(A.get(&m0, N));
        KC_TRY(A.get(&m1, N));
        ::kc::note_launch(), level_morton_keys_k<<<blocks_for(N, 256), 256, 0, s>>>(level, x, d, box, N, m0, v0);
        KC_CUDA(cudaGetLastError());
        KC_TRY(radix_sort_u64_i64(m0, v0, m1, v1, N, 32 + bits_for(h_depth), A, s));
    } else {
        // columns sorted by (level, index)
        uint32_t *k0, *k1;
        KC_TRY(A.get(&k0, N));
        KC_TRY(A.get(&k1, N));
        ::kc::note_launch(), level_keys_k<<<blocks_for(N, 256), 256, 0, s>>>(level, N, k0, v0);
        KC_CUDA(cudaGetLastError());
        KC_TRY(radix_sort_u32_i64(k0, v0, k1, v1, N, bits_for(h_depth), A, s));
    }
    ::kc::note_launch(), order_out_k<<<blocks_for(N, 256), 256, 0, s>>>(v1, N, order);
    KC_CUDA(cudaGetLastError());
    KC_CUDA(cudaStreamSynchronize(s));
    if (depth_out) *depth_out = h_depth;
    return KC_OK;
}

}  // namespace kc
