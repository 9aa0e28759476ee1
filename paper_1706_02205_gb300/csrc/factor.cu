// a5+a6: ICHOL(0) of the Matern kernel matrix restricted to S (Algorithm 2,
// "Incomplete Cholesky factorization with sparsity pattern S"), in its
// left-looking form, as one persistent sync-free kernel.
//
//   for each column i (in dependency order):
//     p    = Theta_ii - sum_{k in R_i} L_ik^2              (FP64)
//     p <= 0  ->  the whole column i is zero (Section 4.4)
//     L_ii = sqrt(p)
//     L_ji = (Theta_ji - sum_{k in R_j cap R_i} L_jk L_ik) / L_ii,  j in C_i
//
// Work units ("tasks") are (column, chunk of up to `rows_per_task` rows of
// C_i), listed in (level, index) order and handed out by an atomic ticket.  A
// team of warps (one, or up to eight for long rows) that takes a task waits
// (bounded, acquire) until every column k in R_i has published all its tasks,
// puts row i (index -> value) into a two-choice hash table in shared memory,
// recomputes the pivot, and then merges the prefix of each row j of its chunk
// (entries k < i) against the table.  The rows of a warp go in batches of 32:
// each lane first fetches one row's bookkeeping and evaluates its Theta_ji from
// the coordinates (entries are never stored), then lanes form groups of G (one
// 32-byte sector of values per group load); a group owns one row, each lane
// walks the row with stride G.  The task publishes by release increments of
// done[i].
//
// Three forms differ in how the prefixes reach the lanes; each lane merges the
// same entries in the same order in all of them, so they give the same bits.
// The ring form (the default) streams them through small shared-memory buffers
// with asynchronous 16-byte copies.  The register form loads U (col, val) pairs
// ahead per lane; it serves other numbers of lanes per row and arrays that do
// not start on a 16-byte boundary.  The bulk form, on request, stages the rows
// of a batch with bulk (TMA) copies into two buffers per warp completing on
// mbarriers; the per-copy cost of the bulk engine for prefixes of a few hundred
// bytes makes it the slowest.
//
// Several independent point sets can be factored in one launch: their
// patterns are concatenated block-diagonally and every column names its set,
// whose Matern parameters the kernel then uses.
//
// FP32 form: values, products and the compensated (Dot2) sums stay in FP32;
// only the pivot and its square root are FP64 (the FP64 pipe of the GB300 is
// a small fraction of its FP32 rate).  FP64 form: everything in FP64.
//
// Forward progress: a task only waits on columns of lower level, whose tasks
// have smaller ticket numbers and were claimed by running warps, so the
// earliest unfinished task can always proceed.  Every wait is bounded: when it
// runs out the kernel records DEV_TIMEOUT in the status word and returns.
#include <algorithm>
#include <type_traits>
#include <vector>

#include "grid.cuh"
#include "ichol.cuh"

namespace kc {

template <typename T>
struct FactorArgs {
    int64_t N;
    int d;
    const double* __restrict__ x;
    const int64_t* __restrict__ rowptr;
    const int32_t* __restrict__ col;
    const int64_t* __restrict__ colptr;
    const int32_t* __restrict__ rowidx;
    const int64_t* __restrict__ slot;
    const int2* __restrict__ tasks;
    const int64_t* __restrict__ ntasks;
    int rpt;  // rows per task
    T* val;
    double* diag;
    unsigned* done;
    unsigned long long* ticket;
    int* status;
    unsigned long long* zero_piv;
    KernelParams kp;                 // kernel of a single set
    const double* __restrict__ aval;  // given entries (ENT = 2): the matrix on the pattern, CSR layout
    const int32_t* __restrict__ col_set;  // set of every column (NULL: one set)
    const KernelParams* __restrict__ kps; // kernels of the sets
    long long spin_limit;
    bool crowded;  // the grid fills the chip
    int hold_col;
    int hbits;  // row table of 2^hbits slots per team
    int lanes;  // lanes per row, 0 = one sector of values
    int adaptive;  // chunk of at least |R_i|/4 rows
    int team;         // warps that share one table (and one task)
    int team_smem;    // shared-memory bytes of one team
    int ctl_off;      // the team's control words within them
    int buf_off;      // the warps' buffers (ring or bulk stages) within them
    int stage_bytes;  // bulk form: bytes of each of the two stage buffers
};

// Rows of column k handled by one task.  Adaptive (on request): at least a
// quarter of |R_k|, because every task re-stages row k, so a long row should
// not be staged again for every few rows below it.
__device__ __forceinline__ int rows_of_task(const int64_t* __restrict__ rowptr, int k, int rpt, int adaptive) {
    if (!adaptive) return rpt;
    const int nr = (int)(rowptr[k + 1] - rowptr[k] - 1);
    return max(rpt, nr >> 2);
}
__device__ __forceinline__ unsigned n_tasks_of(const int64_t* __restrict__ colptr, const int64_t* __restrict__ rowptr,
                                               int k, int rpt, int adaptive) {
    const int64_t m = colptr[k + 1] - colptr[k] - 1;  // rows below the diagonal
    const int r = rows_of_task(rowptr, k, rpt, adaptive);
    return m <= 0 ? 1u : (unsigned)((m + r - 1) / r);
}

// Two-choice table (cuckoo hashing: R. Pagh and F. F. Rodler, J. Algorithms 51
// (2004) 122) of one row i in shared memory: key k in R_i -> L_ik.  A key sits
// in one of the two slots its two hashes name, so a lookup reads at most two
// slots and has no loop: the merges issue the first probes of several entries
// together, then the second ones, which only lanes need whose first slot holds
// another key (a slot once filled stays filled, so an empty first slot means
// the key is absent).  With linear probing the warp walked the probe loops of
// its slowest lane one entry after the other (register form, 2^20 points,
// rho = 3, FP32 form: 45.8 against 41.5 ms).  Empty slots have key -1 and
// value 0; a lookup of key -2 finds nothing.
//
// Insertion moves keys between their two slots.  At the highest load allowed it
// runs out of steps for 3 to 5 % of rows of scattered keys, at 0.9 of that load
// for 0 to 3 %, at half of it for none of thousands (counted for 2^7 to 2^12
// slots); the row is then staged again with other hash multipliers.
constexpr int CK_STEPS = 48;     // moves of one insertion before it gives up
constexpr int CK_TRIES = 4;      // multiplier pairs tried before a row goes without a table
constexpr int CK_LOAD_NUM = 29;  // longest staged row: 29/64 of the slots (a random graph of that many
constexpr int CK_LOAD_DEN = 64;  // edges per vertex stays below the two-choice threshold of 1/2)
__host__ __device__ __forceinline__ int table_rows(int hbits) { return ((1 << hbits) * CK_LOAD_NUM) / CK_LOAD_DEN; }

struct HashPair {
    unsigned m1, m2;  // odd multipliers
    __device__ __forceinline__ explicit HashPair(int attempt = 0)
        : m1(2654435761u + 2u * 0x3C6EF372u * (unsigned)attempt), m2(2246822519u + 2u * 0x1B873593u * (unsigned)attempt) {}
    __device__ __forceinline__ int first(int k, int hbits) const { return (int)(((unsigned)k * m1) >> (32 - hbits)); }
    __device__ __forceinline__ int second(int k, int hbits) const { return (int)(((unsigned)k * m2) >> (32 - hbits)); }
};

// Slots are 8 bytes: the key in the low word and, FP32, the value's bits in
// the high word (a hit needs no further load), FP64, the entry's place in the
// row.  FP64, and tables shared by a team of warps: the row's values lie
// behind the slots in row order (LIN).
template <typename T, bool TEAM>
struct RowTable {
    static constexpr bool INLINE = sizeof(T) == 4;
    static constexpr bool LIN = TEAM || !INLINE;
    unsigned long long* s;
    T* vals;    // LIN: values in row order
    int hbits;  // 2^hbits slots
    HashPair h;
    __device__ __forceinline__ RowTable(unsigned char* base, int hb)
        : s((unsigned long long*)base), vals((T*)(s + (1 << hb))), hbits(hb) {}
    __device__ __forceinline__ void clear(int t, int nt) {
        uint4* q = (uint4*)s;
        for (int i = t; i < (1 << (hbits - 1)); i += nt) q[i] = make_uint4(~0u, 0u, ~0u, 0u);
    }
    // Entry e of the row: key k, value v, by exchanges; false: out of steps
    // (some key is in no slot).  (Storing every entry to its first slot and
    // moving only those that lost theirs was slower: 5.3 against 4.3 ms for
    // 100,003 points in the FP32 form.)
    __device__ __forceinline__ bool insert(int k, int e, T v) {
        unsigned hi;
        if constexpr (INLINE) hi = __float_as_uint(v);
        else hi = (unsigned)e;
        if constexpr (LIN) vals[e] = v;
        unsigned long long w = ((unsigned long long)hi << 32) | (unsigned)k;
        int at = h.first(k, hbits);
        for (int step = 0; step < CK_STEPS; ++step) {
            w = atomicExch(&s[at], w);
            const int out = (int)(unsigned)w;
            if (out < 0) return true;
            const int a1 = h.first(out, hbits);
            at = at == a1 ? h.second(out, hbits) : a1;
        }
        return false;
    }
    // The slots that hold the keys k[], or (another key in the low word) the
    // news that they are absent: PROBES lookups whose loads overlap.
    static constexpr int PROBES = 4;
    __device__ __forceinline__ void probe(const int (&k)[PROBES], unsigned long long (&x)[PROBES]) const {
#pragma unroll
        for (int u = 0; u < PROBES; ++u) x[u] = s[h.first(k[u], hbits)];
#pragma unroll
        for (int u = 0; u < PROBES; ++u) {
            const int key = (int)(unsigned)x[u];
            const unsigned long long* at = &s[h.second(k[u], hbits)];
            if (key != k[u] && key >= 0) x[u] = *at;
        }
    }
    static __device__ __forceinline__ float value(unsigned long long x) { return __uint_as_float((unsigned)(x >> 32)); }
    // acc += L_jk L_ik over the U entries (k[u], w[u]) whose key is in the row.
    // FP32: a miss adds 0 * L_ik', which changes no bit of the sums (the row's
    // values are finite where a column is kept: its pivot holds their squares).
    template <int U>
    __device__ __forceinline__ void merge(const int (&k)[U], const T (&w)[U], Acc<T>& acc) const {
#pragma unroll
        for (int u0 = 0; u0 < U; u0 += PROBES) {
            int kk[PROBES];
            unsigned long long x[PROBES];
#pragma unroll
            for (int u = 0; u < PROBES; ++u) kk[u] = k[u0 + u];
            probe(kk, x);
            if constexpr (INLINE) {
#pragma unroll
                for (int u = 0; u < PROBES; ++u)
                    acc.add((int)(unsigned)x[u] == kk[u] ? w[u0 + u] : 0.f, value(x[u]));
            } else {
                T v[PROBES];
#pragma unroll
                for (int u = 0; u < PROBES; ++u) v[u] = (int)(unsigned)x[u] == kk[u] ? vals[(int)(x[u] >> 32)] : (T)0;
#pragma unroll
                for (int u = 0; u < PROBES; ++u)
                    if ((int)(unsigned)x[u] == kk[u]) acc.add(w[u0 + u], v[u]);  // the FP64 pipe is scarce: hits only
            }
        }
    }
};
// bytes of one table
template <typename T>
static size_t table_bytes(int hbits, bool team) {
    const size_t b = (size_t)8 << hbits;
    const size_t lin = sizeof(T) == 4 && !team ? 0 : sizeof(T) * (size_t)table_rows(hbits);
    return (b + lin + 15) / 16 * 16;
}

// The warps that share one table and work on one task together: a single warp
// where a row's table is small, up to all eight of a CTA for the long rows of
// 3-D patterns, whose tables (8 to 48 KB) would otherwise leave a few warps
// per SM (131,071 points of the cube, rho = 4, FP32 form: 189 ms with a table
// per warp and 12 warps per SM, 73 ms with teams and 24).
struct TeamCtl {
    long long t;  // the task
    int bad;      // 1: a wait ran out, 2: an insertion ran out of steps
};
template <bool TEAM>
struct Team {
    int w = 0, n = 1, bar = 0;
    TeamCtl* ctl = nullptr;
    __device__ __forceinline__ void sync() const {
        if constexpr (TEAM) asm volatile("bar.sync %0, %1;" ::"r"(bar), "r"(32 * n) : "memory");
        else __syncwarp();
    }
};

__device__ __forceinline__ int64_t bsearch_glob(const int32_t* __restrict__ a, int64_t lo, int64_t hi, int k) {
    int64_t end = hi;
    while (lo < hi) {
        int64_t mid = (lo + hi) >> 1;
        if (__ldg(&a[mid]) < k) lo = mid + 1;
        else hi = mid;
    }
    return (lo < end && __ldg(&a[lo]) == k) ? lo : -1;
}

// Matern parameters of column i's set, read where they are used (not kept in
// registers through the merges).
template <typename T>
__device__ __forceinline__ const KernelParams& kparams(const FactorArgs<T>& A, int i) {
    return A.col_set ? A.kps[A.col_set[i]] : A.kp;
}

// Everything a warp knows of its task.
template <typename T>
struct TaskCtx {
    int i, c, nr;
    int64_t a0;      // R_i = col[a0 .. a0 + nr), L_ii at a0 + nr
    int64_t qs, qe;  // the warp's rows of the column: CSC positions
    bool zero;       // dropped pivot: the whole column is zero
    bool staged;     // row i is in the table (else binary search in global memory)
    double Lii;
    T inv;
};

// An insertion of row i ran out of steps: stage the row (nr entries at col,
// val, its columns complete by now) again with other multipliers.  Returns the
// attempt that succeeded, or 0: the row goes without a table.
template <typename T, bool TEAM>
__device__ __noinline__ int restage(RowTable<T, TEAM> tab, Team<TEAM> tm, const int32_t* col, const T* val, int nr) {
    const int lane = lane_id();
    for (int attempt = 1; attempt < CK_TRIES; ++attempt) {
        tab.h = HashPair(attempt);
        tm.sync();
        if constexpr (TEAM) {
            if (tm.w == 0 && lane == 0) tm.ctl->bad = 0;
        }
        tab.clear(32 * tm.w + lane, 32 * tm.n);
        tm.sync();
        bool placed = true;
        for (int e = 32 * tm.w + lane; e < nr; e += 32 * tm.n) placed &= tab.insert(col[e], e, ldcg(val + e));
        if constexpr (TEAM) {
            if (!placed) tm.ctl->bad = 2;
            tm.sync();
            if (*(volatile int*)&tm.ctl->bad == 0) return attempt;
        } else {
            if (__all_sync(0xffffffffu, placed)) return attempt;
        }
    }
    tm.sync();  // every warp has read `bad` before the first one claims another task and clears it
    return 0;
}

// Claim the next task.  False: no tasks left, or the kernel is stopping.
template <typename T, bool TEAM>
__device__ __forceinline__ bool task_claim(const FactorArgs<T>& A, const Team<TEAM>& tm, int rows_round, int lane,
                                           TaskCtx<T>& X) {
    int64_t t = 0;
    if constexpr (TEAM) {
        if (tm.w == 0 && lane == 0) {
            t = (int64_t)atomicAdd(A.ticket, 1ULL);
            tm.ctl->t = t >= __ldg(A.ntasks) || ld_volatile_s32(A.status) != 0 ? -1 : t;
            tm.ctl->bad = 0;
        }
        tm.sync();  // also: every warp of the team is done with the previous task's table
        t = *(volatile long long*)&tm.ctl->t;
        if (t < 0) return false;
    } else {
        if (lane == 0) t = (int64_t)atomicAdd(A.ticket, 1ULL);
        t = __shfl_sync(0xffffffffu, t, 0);
        if (t >= __ldg(A.ntasks) || ld_volatile_s32(A.status) != 0) return false;
    }
    const int2 tk = A.tasks[t];
    X.i = tk.x;
    X.c = tk.y;
    X.a0 = A.rowptr[X.i];
    X.nr = (int)(A.rowptr[X.i + 1] - 1 - X.a0);
    const int rows = rows_of_task(A.rowptr, X.i, A.rpt, A.adaptive);
    X.qs = A.colptr[X.i] + 1 + (int64_t)X.c * rows;
    X.qe = min(A.colptr[X.i + 1], X.qs + rows);
    if constexpr (TEAM) {  // the warp's share, in whole rounds of rows
        const int per = ((int)(X.qe - X.qs) + rows_round * tm.n - 1) / (rows_round * tm.n) * rows_round;
        X.qs += (int64_t)tm.w * per;
        X.qe = min(X.qe, X.qs + per);
    }
    return true;
}

// The prologue of a task: wait until every column k in R_i is complete, put
// row i into the table, form the pivot in FP64.  `ready` runs as soon as the
// columns are known to be complete (their values may be read), beside the
// table and the pivot.  False: a wait ran out or the kernel is stopping.
template <typename T, int ENT, bool TEAM, typename Ready>
__device__ __forceinline__ bool task_stage(const FactorArgs<T>& A, const Team<TEAM>& tm, RowTable<T, TEAM>& tab,
                                           int lane, TaskCtx<T>& X, Ready&& ready) {
    const unsigned FULL = 0xffffffffu;
    X.staged = X.nr <= table_rows(A.hbits);
    tab.h = HashPair();
    if (X.staged) tab.clear(32 * tm.w + lane, 32 * tm.n);
    tm.sync();
    // R_i in rounds of DEPS entries per lane: the column indices, the completion
    // counters of those columns (await_columns), one acquire fence, then
    // the values into the table and, for a single warp, the sum of squares (the
    // accumulator of the merges: FP32 form compensated, its two parts added in
    // FP64 below).  Each lane reads only the values of the columns it checked
    // itself; the other lanes' columns are ordered by the barrier after that.
    constexpr int DEPS = 8;
    Acc<T> sq;
    bool placed = true, ok = true;
    const int step = 32 * tm.n;
    for (int first = 0; first < X.nr || first == 0; first += step * DEPS) {
        const int e0 = first + 32 * tm.w + lane;
        int kk[DEPS];
#pragma unroll
        for (int u = 0; u < DEPS; ++u) kk[u] = e0 + step * u < X.nr ? __ldg(&A.col[X.a0 + e0 + step * u]) : -1;
        // A team keeps a failure until its rounds are over (leaving the loop at once costs it registers:
        // 8 bytes more of spills, 0.9 % of 131,071 points of the cube); a single warp leaves below.
        if constexpr (TEAM) ok &= await_columns<DEPS>(A.done, kk, A.status, A.spin_limit, A.crowded);
        else ok = await_columns<DEPS>(A.done, kk, A.status, A.spin_limit, A.crowded);
        fence_acq_rel_gpu();  // acquire: the columns' values are visible from here on
        if (!ok)
#pragma unroll
            for (int u = 0; u < DEPS; ++u) kk[u] = -1;
        T vv[DEPS];
#pragma unroll
        for (int u = 0; u < DEPS; ++u) vv[u] = kk[u] >= 0 ? ldcg(&A.val[X.a0 + e0 + step * u]) : (T)0;
        if constexpr (!TEAM) {
            __syncwarp();
            if (ok && first + step * DEPS >= X.nr) ready();
        }
        if (X.staged) {
#pragma unroll
            for (int u = 0; u < DEPS; ++u)
                if (kk[u] >= 0) placed &= tab.insert(kk[u], e0 + step * u, vv[u]);
        }
        if constexpr (!TEAM) {
#pragma unroll
            for (int u = 0; u < DEPS; ++u)
                if (kk[u] >= 0) sq.add(vv[u], vv[u]);
        }
        if constexpr (!TEAM) {
            if (!ok) break;
        }
    }
    if constexpr (TEAM) {
        if (!ok || !placed) atomicOr(&tm.ctl->bad, ok ? 2 : 1);
        tm.sync();  // the table and the row's values are complete
        const int bad = *(volatile int*)&tm.ctl->bad;
        if (bad & 1) {
            if (lane == 0) atomicCAS(A.status, 0, DEV_TIMEOUT);
            return false;
        }
        placed = bad == 0;
        ready();
    } else {
        if (!ok) {
            if (lane == 0) atomicCAS(A.status, 0, DEV_TIMEOUT);
            return false;
        }
        placed = __all_sync(FULL, placed);
    }
    if (!placed) {
        const int attempt = restage<T, TEAM>(tab, tm, A.col + X.a0, A.val + X.a0, X.nr);
        tab.h = HashPair(attempt);
        X.staged = attempt > 0;
    }
    if constexpr (TEAM) {  // every warp forms the pivot, each lane over the entries a single warp's lane would take
        for (int e = lane; e < X.nr; e += 32) {
            const T v = X.staged ? tab.vals[e] : ldcg(&A.val[X.a0 + e]);
            sq.add(v, v);
        }
    }
    sq.group_reduce(32);
    // Lane 0 forms the pivot and every lane takes its values: one pivot for the
    // whole task whichever lane writes a row (after a butterfly the partners'
    // compensations c + (c2 + e) and c2 + (c + e) may round apart), and the FP64
    // work runs on one lane.
    double Lii = 0.0;
    T inv = (T)0;
    int zero = 0;
    if (lane == 0) {
        const int64_t a1 = X.a0 + X.nr;
        double thii;
        if constexpr (ENT == 2) {
            thii = A.aval[a1];
        } else {
            const KernelParams& kp = kparams(A, X.i);
            thii = kp.sigma2 + kp.nugget;
        }
        const double p = thii - sq.total();
        zero = !(p > 0.0);
        Lii = zero ? 0.0 : sqrt(p);
        inv = zero ? (T)0 : Acc<T>::recip(Lii);
        if (X.c == 0 && tm.w == 0) {
            A.val[a1] = (T)Lii;
            A.diag[X.i] = Lii;
            if (zero) atomicAdd(A.zero_piv, 1ULL);
        }
    }
    X.Lii = __shfl_sync(FULL, Lii, 0);
    X.inv = __shfl_sync(FULL, inv, 0);
    X.zero = __shfl_sync(FULL, zero, 0) != 0;
    __syncwarp();  // a single warp: the table's inserts are visible to every lane
    return true;
}

// Publish the warp's part of a finished task of column i: its lanes' writes,
// ordered before lane 0's fence by the warp barrier, then the count.
template <typename T>
__device__ __forceinline__ void task_end(const FactorArgs<T>& A, int i, int lane) {
    __syncwarp();
    if (lane == 0 && i != A.hold_col) {
        fence_acq_rel_gpu();
        red_release_add_u32(&A.done[i], 1u);
    }
}

// Lanes per row: one 32-byte sector of values per group load (8 lanes in
// FP32, 4 in FP64), unless set.
template <typename T>
__device__ __forceinline__ int lanes_per_row(int lanes) {
    return lanes > 0 ? lanes : (int)(32 / sizeof(T));
}

// Merge of the prefix [es, be) of row j, read from global memory, against
// row i: U (col, val) pairs per lane in flight; the ragged end is masked.
template <typename T, int U, bool TEAM>
__device__ __forceinline__ void merge_global(const FactorArgs<T>& A, const RowTable<T, TEAM>& tab, const TaskCtx<T>& X,
                                             int64_t es, int64_t be, int sub, int G, Acc<T>& acc) {
    if (X.staged) {
        const int n = (int)(be - es);
        const int32_t* cp = A.col + es;
        const T* vp = A.val + es;
        for (int t = sub; t < n; t += U * G) {
            int k[U];
            T wv[U];
#pragma unroll
            for (int u = 0; u < U; ++u) k[u] = t + u * G < n ? __ldg(cp + t + u * G) : -2;
#pragma unroll
            for (int u = 0; u < U; ++u) wv[u] = t + u * G < n ? ldcg(vp + t + u * G) : (T)0;
            tab.template merge<U>(k, wv, acc);
        }
    } else {
        for (int64_t e = es + sub; e < be; e += G) {
            const int64_t pos = bsearch_glob(A.col, X.a0, X.a0 + X.nr, __ldg(&A.col[e]));
            if (pos >= 0) acc.add(ldcg(&A.val[e]), ldcg(&A.val[pos]));
        }
    }
}

// Row-j bookkeeping of the rows b0+lane of a batch: the slot of L_ji, the
// start of row j, and Theta_ji (loads and exponentials overlap across lanes).
// None of it depends on other columns, so the first batch's is fetched before
// the task waits for them.
template <typename T, int ENT>
__device__ __forceinline__ void batch_rows(const FactorArgs<T>& A, int i, int64_t b0, int nb, int lane,
                                           int64_t& my_e0, int64_t& my_b, T& my_th) {
    my_e0 = 0;
    my_b = 0;
    my_th = (T)0;
    if (lane < nb) {
        const int j = __ldg(&A.rowidx[b0 + lane]);
        my_b = __ldg(&A.slot[b0 + lane]);
        my_e0 = __ldg(&A.rowptr[j]);
        if constexpr (ENT == 2)
            my_th = (T)__ldg(&A.aval[my_b]);
        else
            my_th = theta_off<T, ENT == 1>(kparams(A, i), A.d, A.x + (int64_t)j * A.d, A.x + (int64_t)i * A.d);
    }
}

// The team, its table and its control words.
template <typename T, bool TEAM>
__device__ __forceinline__ Team<TEAM> make_team(const FactorArgs<T>& A, unsigned char* smem, int warp,
                                                unsigned char** base) {
    Team<TEAM> tm;
    int q = warp;
    if constexpr (TEAM) {
        q = warp / A.team;
        tm.w = warp % A.team;
        tm.n = A.team;
        tm.bar = 1 + q;
    }
    *base = smem + (size_t)q * A.team_smem;
    if constexpr (TEAM) tm.ctl = (TeamCtl*)(*base + A.ctl_off);
    return tm;
}

// --------------------------------------------------------------- ring form
// The default.  The row prefixes of a batch flow through a ring of RING
// shared-memory buffers per warp: in every step each group of G lanes merges
// CH entries of its row from one buffer while the copies of the next RING - 1
// steps are in flight (cp.async, 16 bytes a lane, straight from L2 to shared
// memory).  The bytes in flight cost no registers and never drain between
// rows: with the loads in registers a warp waited a full memory latency in
// every round of rows (issue slots 52 % busy; now 64 %).  A 16-byte copy must
// start on a 16-byte boundary, so a row's copies start up to 3 entries before
// its prefix; those entries are masked, and what lies behind the prefix is
// copied as zeros.  Each lane takes the same entries in the same order as in
// the register form, so both give the same bits.
//
// Measured at 2^20 points, rho = 3, FP32 form (151 GB of operand stream, 22 ms
// at the copy rate): 35.8 ms; register form with the same table 41.5, with a
// linear-probing table 45.8.  Ring of 3, 4, 5, 6, 8 buffers: 40.2, 38.0, 38.8,
// 39.8, 41.2 (before the grid rule below).  16, 32, 64 entries a step: 44.8
// (two rows a lane, packed FP32x2 sums), 38.0, 42.5.  Bound now by issue slots,
// shared-memory wavefronts (60 %) and HBM (59 % of the copy rate) alike.
constexpr int RING = 4;

template <typename T>
struct RingLayout {
    static constexpr int G = 32 / (int)sizeof(T);  // lanes per row
    static constexpr int RR = 32 / G;              // rows per step
    static constexpr int SL = 4;                   // entries per lane and step
    static constexpr int CH = SL * G;              // entries per row and step
    static constexpr int COLB = RR * CH * 4, VALB = RR * CH * (int)sizeof(T);
    static constexpr int STAGE = COLB + VALB;
    // First place of block blk (G entries) of row r: the blocks of a row are
    // rotated by row so that the reads of a step fall into different banks.
    static __device__ __forceinline__ int col_at(int r, int blk) {
        return r * CH + ((blk + (sizeof(T) == 8 ? r >> 1 : r)) & (SL - 1)) * G;
    }
    static __device__ __forceinline__ int val_at(int r, int blk) { return r * CH + ((blk + r) & (SL - 1)) * G; }
};

__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
// 16-byte copy of which the first `bytes` are read and the rest is zero
__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src, int bytes) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// Resident CTAs of 8 warps per SM that the register budget is cut for.
#ifndef KC_FACTOR_MIN_BLOCKS
#define KC_FACTOR_MIN_BLOCKS 4
#endif

template <typename T, int ENT, bool TEAM>
__global__ void __launch_bounds__(256, 3) ichol_ring_k(FactorArgs<T> A) {
    using RL = RingLayout<T>;
    constexpr int G = RL::G, RR = RL::RR, CH = RL::CH, SL = RL::SL;
    extern __shared__ __align__(16) unsigned char smem[];
    const int lane = lane_id();
    const unsigned FULL = 0xffffffffu;
    unsigned char* base;
    const Team<TEAM> tm = make_team<T, TEAM>(A, smem, threadIdx.x >> 5, &base);
    RowTable<T, TEAM> tab(base, A.hbits);
    unsigned char* ring = base + A.buf_off + (size_t)tm.w * (RING * RL::STAGE);
    const int g = lane / G, sub = lane % G;
    // the lane's copies of one step: 4 entries of its group's row, from the (4 sub)-th on
    const uint32_t rs = smem_addr(ring);
    const uint32_t dcol = rs + 4u * (uint32_t)(RL::col_at(g, 4 * sub / G) + 4 * sub % G);
    const uint32_t dval = rs + RL::COLB + (uint32_t)sizeof(T) * (uint32_t)(RL::val_at(g, 4 * sub / G) + 4 * sub % G);
    TaskCtx<T> X{};
    unsigned in_st = 0, out_st = 0;  // ring buffers to fill and to merge next
    // the batch: the lane's row (L_ji at my_b, its prefix from my_e0 on, Theta_ji), its entries with the leading
    // ones of its first copy, and the steps of the longest row of its round
    int64_t my_e0, my_b;
    T my_th;
    int nb, my_n, steps;
    // the filling end of the ring: `left` steps of the round from row pr on; of the group's row `n` entries from the
    // lane's first one on
    int pr, left, n;
    const int32_t* cp = A.col;
    const T* vp = A.val;
    auto batch = [&](int64_t b0) {
        nb = (int)max((int64_t)0, min((int64_t)32, X.qe - b0));
        batch_rows<T, ENT>(A, X.i, b0, nb, lane, my_e0, my_b, my_th);
        my_n = (int)(my_b - (my_e0 & ~(int64_t)3));
        steps = max(1, (my_n + CH - 1) / CH);
#pragma unroll
        for (int o = 1; o < RR; o <<= 1) steps = max(steps, __shfl_xor_sync(FULL, steps, o));
        pr = -RR;
        left = n = 0;
    };
    auto fill = [&]() {
        if (left == 0) {
            pr += RR;
            if (pr < nb) {
                const int64_t es = (__shfl_sync(FULL, my_e0, pr + g) & ~(int64_t)3) + 4 * sub;
                n = __shfl_sync(FULL, my_n, pr + g) - 4 * sub;
                left = __shfl_sync(FULL, steps, pr);
                cp = A.col + es;
                vp = A.val + es;
            }
        }
        if (left > 0) {
            const uint32_t off = in_st * (uint32_t)RL::STAGE;
            cp_async16(dcol + off, cp, max(0, min(16, 4 * n)));
            if constexpr (sizeof(T) == 4) {
                cp_async16(dval + off, vp, max(0, min(16, 4 * n)));
            } else {
                cp_async16(dval + off, vp, max(0, min(16, 8 * n)));
                cp_async16(dval + off + 16, vp + 2, max(0, min(16, 8 * (n - 2))));
            }
            cp += CH;
            vp += CH;
            n -= CH;
            --left;
            in_st = (in_st + 1) % RING;
        }
        cp_async_commit();
    };
    auto start = [&]() {
#pragma unroll
        for (int q = 0; q < RING - 1; ++q) fill();
    };
    for (;;) {
        if (!task_claim<T, TEAM>(A, tm, RR, lane, X)) break;
        batch(X.qs);
        if (!task_stage<T, ENT, TEAM>(A, tm, tab, lane, X, start)) break;
        if (X.zero || !X.staged) {  // the copies are not used
            cp_async_wait<0>();
            in_st = out_st = 0;
        }
        for (int64_t b0 = X.qs; b0 < X.qe; b0 += 32) {
            if (b0 != X.qs) {
                batch(b0);
                if (!X.zero && X.staged) start();
            }
            if (X.zero || !X.staged) {  // dropped column; row i without a table
                for (int r0 = 0; r0 < nb; r0 += RR) {
                    const int r = r0 + g;
                    const int64_t es = __shfl_sync(FULL, my_e0, r & 31), be = __shfl_sync(FULL, my_b, r & 31);
                    const T th = __shfl_sync(FULL, my_th, r & 31);
                    Acc<T> acc;
                    if (r < nb && !X.zero) merge_global<T, 4, TEAM>(A, tab, X, es, be, sub, G, acc);
                    acc.group_reduce(G);
                    if (r < nb && sub == 0) A.val[be] = X.zero ? (T)0 : acc.finish(th, X.Lii, X.inv);
                }
                continue;
            }
            for (int r0 = 0; r0 < nb; r0 += RR) {
                const int m = __shfl_sync(FULL, steps, r0);
                const int r = r0 + g;
                // The row's prefix starts sh entries into its copies.  The lane's entries, the sub-th of the prefix and
                // every G-th after it, lie at place x of each block; where x < sh the first block's is not of the row.
                const int sh = (int)__shfl_sync(FULL, (unsigned)my_e0, r) & 3;
                const int x = (sub + sh) % G;
                bool before = x < sh;
                // FP64: the padding behind the prefix is kept off the FP64 pipe
                [[maybe_unused]] int rest = __shfl_sync(FULL, my_n, r) - x;
                Acc<T> acc;
                for (int c = 0; c < m; ++c) {
                    cp_async_wait<RING - 2>();
                    __syncwarp();  // the step's copies of every lane have landed, and the buffer filled next is free
                    const int* kc_ = (const int*)(ring + out_st * RL::STAGE) + x;
                    const T* vc = (const T*)(ring + out_st * RL::STAGE + RL::COLB) + x;
                    int k[SL];
                    T w[SL];
#pragma unroll
                    for (int v = 0; v < SL; ++v) {
                        k[v] = kc_[RL::col_at(g, v)];
                        w[v] = vc[RL::val_at(g, v)];
                    }
                    fill();
                    if (before) k[0] = -2;
                    before = false;
                    if constexpr (sizeof(T) == 8) {
#pragma unroll
                        for (int v = 0; v < SL; ++v)
                            if (v * G >= rest) k[v] = -2;
                        rest -= CH;
                    }
                    tab.template merge<SL>(k, w, acc);
                    out_st = (out_st + 1) % RING;
                }
                acc.group_reduce(G);
                const int64_t be = __shfl_sync(FULL, my_b, r);
                const T th = __shfl_sync(FULL, my_th, r);
                if (r < nb && sub == 0) A.val[be] = acc.finish(th, X.Lii, X.inv);
            }
        }
        task_end(A, X.i, lane);
    }
    cp_async_wait<0>();
}

// ----------------------------------------------------------- register form
// Each lane keeps U (col, val) loads of its row prefix in flight in registers.
// Taken for another number of lanes per row than the ring's, and for values or
// column indices that do not start on a 16-byte boundary.
template <typename T, int U, int ENT, bool TEAM>
__global__ void __launch_bounds__(256, U >= 16 ? 3 : KC_FACTOR_MIN_BLOCKS) ichol_persistent_k(FactorArgs<T> A) {
    extern __shared__ __align__(16) unsigned char smem[];
    const int lane = lane_id();
    const unsigned FULL = 0xffffffffu;
    unsigned char* base;
    const Team<TEAM> tm = make_team<T, TEAM>(A, smem, threadIdx.x >> 5, &base);
    RowTable<T, TEAM> tab(base, A.hbits);
    TaskCtx<T> X{};
    const int G = lanes_per_row<T>(A.lanes);
    const int ng = 32 / G, g = lane / G, sub = lane % G;
    for (;;) {
        if (!task_claim<T, TEAM>(A, tm, ng, lane, X)) return;
        if (!task_stage<T, ENT, TEAM>(A, tm, tab, lane, X, [] {})) return;
        for (int64_t b0 = X.qs; b0 < X.qe; b0 += 32) {
            const int nb = (int)min((int64_t)32, X.qe - b0);
            int64_t my_e0, my_b;
            T my_th;
            batch_rows<T, ENT>(A, X.i, b0, nb, lane, my_e0, my_b, my_th);
            for (int r0 = 0; r0 < nb; r0 += ng) {
                const int r = r0 + g;
                const bool act = r < nb;
                const int src = act ? r : 0;
                const int64_t es = __shfl_sync(FULL, my_e0, src);
                const int64_t be = __shfl_sync(FULL, my_b, src);  // L_ji lives at be; the prefix is [es, be)
                const T th = __shfl_sync(FULL, my_th, src);
                Acc<T> acc;
                if (act && !X.zero) merge_global<T, U, TEAM>(A, tab, X, es, be, sub, G, acc);
                acc.group_reduce(G);
                if (act && sub == 0) A.val[be] = X.zero ? (T)0 : acc.finish(th, X.Lii, X.inv);
            }
        }
        task_end(A, X.i, lane);
    }
}

// --------------------------------------------------------------- bulk form
// The prefixes of a stage of consecutive rows are copied from global memory
// into one of two shared-memory buffers of the warp by the bulk-copy (TMA)
// engine, completing on an mbarrier; the warp merges the previous stage from
// shared memory meanwhile.  The loads in flight then cost no registers, so a
// few warps per SM keep enough bytes in flight.  Each row's (col, val)
// extents are widened to 16-byte boundaries (a bulk copy's rule); a row that
// alone exceeds a buffer is merged from global memory instead.
__device__ __forceinline__ void mbar_init(uint64_t* bar) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(bar)) : "memory");
}
__device__ __forceinline__ void mbar_expect(uint64_t* bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)), "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ bool mbar_test(uint64_t* bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_addr(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}
// bounded wait for the phase with the given parity to complete
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, long long limit) {
    if (mbar_test(bar, parity)) return true;
    const long long t0 = clock64();
    while (!mbar_test(bar, parity))
        if (clock64() - t0 > limit) return false;
    return true;
}
__device__ __forceinline__ void bulk_copy(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                     smem_addr(dst)),
                 "l"(src), "r"(bytes), "r"(smem_addr(bar))
                 : "memory");
}

// A stage: rows [s0, s1) of the current batch, in buffer `buf`; `direct`: one
// row merged from global memory; `bytes`: the buffer's barrier is armed.
struct Stage {
    int s0, s1, buf;
    bool direct, bytes;
};

// Issue the copies of the next stage starting at row c0 of the batch into
// buffer bi.  Each lane owns row lane of the batch: it sizes its widened
// extents, a warp scan places them, and the rows that fit are copied.
// my_off / my_meta receive the position of the lane's row in the buffer.
template <typename T>
__device__ __forceinline__ Stage stage_issue(const FactorArgs<T>& A, unsigned char* buf, uint64_t* bar, int bi,
                                             int c0, int nb, int lane, int64_t my_e0, int64_t my_b,
                                             uint32_t& my_off, uint32_t& my_meta) {
    const unsigned FULL = 0xffffffffu;
    uint32_t sz = 0, colB = 0, hc = 0, hv = 0;
    uintptr_t cl = 0, vl = 0;
    const bool mine = lane >= c0 && lane < nb;
    if (mine && my_b > my_e0) {
        const uintptr_t ca = (uintptr_t)(A.col + my_e0), ce = (uintptr_t)(A.col + my_b);
        const uintptr_t va = (uintptr_t)(A.val + my_e0), ve = (uintptr_t)(A.val + my_b);
        cl = ca & ~(uintptr_t)15;
        vl = va & ~(uintptr_t)15;
        colB = (uint32_t)(((ce + 15) & ~(uintptr_t)15) - cl);
        sz = colB + (uint32_t)(((ve + 15) & ~(uintptr_t)15) - vl);
        hc = (uint32_t)((ca - cl) >> 2);
        hv = (uint32_t)((va - vl) / sizeof(T));
    }
    uint32_t inc = sz;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t n = __shfl_up_sync(FULL, inc, o);
        if (lane >= o) inc += n;
    }
    const bool fits = mine && inc <= (uint32_t)A.stage_bytes;
    const int cnt = __popc(__ballot_sync(FULL, fits));  // rows c0 .. c0+cnt-1: the scan is monotone
    Stage S;
    S.s0 = c0;
    S.buf = bi;
    if (cnt == 0) {
        S.s1 = c0 + 1;
        S.direct = true;
        S.bytes = false;
        return S;
    }
    S.s1 = c0 + cnt;
    S.direct = false;
    const uint32_t total = __shfl_sync(FULL, inc, c0 + cnt - 1);
    S.bytes = total > 0;
    if (fits) {
        my_off = inc - sz;
        my_meta = colB | (hc << 24) | (hv << 28);
    }
    if (S.bytes) {
        // the buffer's previous contents were read by this warp's generic loads
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        if (lane == 0) mbar_expect(bar, total);
        __syncwarp();
        if (fits && sz > 0) {
            bulk_copy(buf + (inc - sz), (const void*)cl, colB, bar);
            bulk_copy(buf + (inc - sz) + colB, (const void*)vl, sz - colB, bar);
        }
    }
    return S;
}

// Merge of a prefix of n entries held in shared memory.
template <typename T, int U>
__device__ __forceinline__ void merge_smem(const RowTable<T, false>& tab, const int* cs, const T* vs, int n, int sub, int G,
                                           Acc<T>& acc) {
    for (int t = sub; t < n; t += U * G) {
        int k[U];
        T wv[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int q = t + u * G;
            k[u] = q < n ? cs[q] : -2;
            wv[u] = q < n ? vs[q] : (T)0;
        }
        tab.template merge<U>(k, wv, acc);
    }
}

template <typename T, int U, int ENT>
__global__ void __launch_bounds__(128) ichol_bulk_k(FactorArgs<T> A) {
    extern __shared__ __align__(16) unsigned char smem[];
    const int lane = lane_id();
    const int w = threadIdx.x >> 5;
    unsigned char* base = smem + (size_t)w * A.team_smem;
    RowTable<T, false> tab(base, A.hbits);
    const Team<false> tm;
    unsigned char* bufs = base + A.buf_off;
    uint64_t* bars = (uint64_t*)(bufs + 2 * (size_t)A.stage_bytes);
    const unsigned FULL = 0xffffffffu;
    if (lane == 0) {
        mbar_init(&bars[0]);
        mbar_init(&bars[1]);
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    __syncwarp();
    uint32_t phase = 0;  // bit b: parity of the next phase of barrier b
    TaskCtx<T> X{};
    for (;;) {
        if (!task_claim<T, false>(A, tm, 1, lane, X)) return;
        if (!task_stage<T, ENT, false>(A, tm, tab, lane, X, [] {})) return;
        // values of finished columns were written by other SMs through the generic
        // proxy and acquired above; the bulk copies read them through the async proxy
        asm volatile("fence.proxy.async.global;" ::: "memory");
        const int G = lanes_per_row<T>(A.lanes);
        const int ng = 32 / G, g = lane / G, sub = lane % G;
        const bool bulk = X.staged && !X.zero;
        for (int64_t b0 = X.qs; b0 < X.qe; b0 += 32) {
            const int nb = (int)min((int64_t)32, X.qe - b0);
            int64_t my_e0, my_b;
            T my_th;
            batch_rows<T, ENT>(A, X.i, b0, nb, lane, my_e0, my_b, my_th);
            uint32_t off0 = 0, meta0 = 0, off1 = 0, meta1 = 0;  // the lane's row in buffer 0 / 1
            Stage cur;
            if (bulk) cur = stage_issue(A, bufs, &bars[0], 0, 0, nb, lane, my_e0, my_b, off0, meta0);
            else cur = Stage{0, nb, 0, true, false};
            while (cur.s0 < nb) {
                Stage nxt{nb, nb, 0, true, false};
                if (bulk && cur.s1 < nb) {
                    if (cur.buf == 0)
                        nxt = stage_issue(A, bufs + A.stage_bytes, &bars[1], 1, cur.s1, nb, lane, my_e0, my_b, off1,
                                          meta1);
                    else
                        nxt = stage_issue(A, bufs, &bars[0], 0, cur.s1, nb, lane, my_e0, my_b, off0, meta0);
                }
                if (cur.bytes) {
                    const bool ok = mbar_wait(&bars[cur.buf], (phase >> cur.buf) & 1u, A.spin_limit);
                    phase ^= 1u << cur.buf;
                    if (!__all_sync(FULL, ok)) {
                        // give the copies still in flight a bounded chance to land, then stop
                        if (nxt.bytes) mbar_wait(&bars[nxt.buf], (phase >> nxt.buf) & 1u, A.spin_limit);
                        if (lane == 0) atomicCAS(A.status, 0, DEV_TIMEOUT);
                        return;
                    }
                }
                const unsigned char* sb = bufs + (size_t)cur.buf * A.stage_bytes;
                const uint32_t my_off = cur.buf ? off1 : off0, my_meta = cur.buf ? meta1 : meta0;
                for (int r0 = cur.s0; r0 < cur.s1; r0 += ng) {
                    const int r = r0 + g;
                    const bool act = r < cur.s1;
                    const int src = act ? r : cur.s0;
                    const int64_t es = __shfl_sync(FULL, my_e0, src);
                    const int64_t be = __shfl_sync(FULL, my_b, src);
                    const T th = __shfl_sync(FULL, my_th, src);
                    const uint32_t ro = __shfl_sync(FULL, my_off, src);
                    const uint32_t rm = __shfl_sync(FULL, my_meta, src);
                    Acc<T> acc;
                    if (act && !X.zero) {
                        if (cur.direct) {
                            merge_global<T, U, false>(A, tab, X, es, be, sub, G, acc);
                        } else {
                            const uint32_t colB = rm & 0xffffffu;
                            const int* cs = (const int*)(sb + ro) + (rm >> 24 & 15u);
                            const T* vs = (const T*)(sb + ro + colB) + (rm >> 28);
                            merge_smem<T, U>(tab, cs, vs, (int)(be - es), sub, G, acc);
                        }
                    }
                    acc.group_reduce(G);
                    if (act && sub == 0) A.val[be] = X.zero ? (T)0 : acc.finish(th, X.Lii, X.inv);
                }
                __syncwarp();
                cur = nxt;
            }
        }
        task_end(A, X.i, lane);
    }
}

// done[k] = -(tasks of column k) * (warps that publish each), as an unsigned word
__global__ void done_init_k(const int64_t* __restrict__ colptr, const int64_t* __restrict__ rowptr, int64_t N, int rpt,
                            int adaptive, int team, unsigned* __restrict__ done) {
    int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (k < N) done[k] = 0u - n_tasks_of(colptr, rowptr, (int)k, rpt, adaptive) * (unsigned)team;
}

// tasks of column order[p]: n_tasks_of(order[p])
__global__ void task_count_k(const int32_t* __restrict__ order, const int64_t* __restrict__ colptr,
                             const int64_t* __restrict__ rowptr, int64_t N, int rpt, int adaptive,
                             int64_t* __restrict__ cnt) {
    int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p < N) cnt[p] = n_tasks_of(colptr, rowptr, order[p], rpt, adaptive);
}
__global__ void task_fill_k(const int32_t* __restrict__ order, const int64_t* __restrict__ toff, int64_t N,
                            int2* __restrict__ tasks) {
    int64_t p = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    int lane = lane_id();
    if (p < N) {
        int64_t a = toff[p], b = toff[p + 1];
        int i = order[p];
        for (int64_t t = a + lane; t < b; t += 32) tasks[t] = make_int2(i, (int)(t - a));
    }
}
__global__ void max_row_k(const int64_t* __restrict__ rowptr, int64_t N, int* __restrict__ out) {
    int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    int m = 0;
    if (j < N) m = (int)(rowptr[j + 1] - rowptr[j] - 1);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
    if (lane_id() == 0) atomicMax(out, m);
}

// Longest row of L without its diagonal (synchronises).
static kc_status max_row(const kc_pattern* P, Arena& A, cudaStream_t s, int* out) {
    int* mr;
    KC_TRY(A.get(&mr, 1));
    KC_CUDA(cudaMemsetAsync(mr, 0, sizeof(int), s));
    ::kc::note_launch(), max_row_k<<<blocks_for(P->N, 256), 256, 0, s>>>(P->rowptr, P->N, mr);
    KC_CUDA(cudaGetLastError());
    KC_CUDA(cudaMemcpyAsync(out, mr, sizeof(int), cudaMemcpyDeviceToHost, s));
    KC_CUDA(cudaStreamSynchronize(s));
    return KC_OK;
}

// Tasks a pattern has at most: one per column and one more per rpt rows below the diagonal.
int64_t tasks_bound(const kc_pattern* P, int rpt) { return P->N + (P->nnz - P->N) / rpt; }

// Build the task list of a pattern (its columns in the schedule's order:
// by level, within a level in space-filling-curve order when the schedule was
// given the points, so that consecutive tasks merge rows of neighbouring
// points, which share most of their entries).  The count stays on the device
// (*count_out); with ntasks_out it also goes to the host, which waits for it.
kc_status build_tasks(const kc_pattern* P, int rpt, Arena& A, cudaStream_t s, int2** tasks_out,
                      const int64_t** count_out, int64_t* ntasks_out, bool adaptive) {
    int64_t N = P->N;
    int64_t* cnt;
    int64_t* toff;
    KC_TRY(A.get(&cnt, N));
    KC_TRY(A.get(&toff, N + 1));
    const int32_t* order = P->order;
    ::kc::note_launch(), task_count_k<<<blocks_for(N, 256), 256, 0, s>>>(order, P->colptr, P->rowptr, N, rpt,
                                                                            adaptive ? 1 : 0, cnt);
    KC_TRY(exclusive_scan_i64(cnt, toff, N, A, s));
    KC_CUDA(cudaGetLastError());
    int64_t nt = tasks_bound(P, rpt);
    if (ntasks_out) {
        KC_CUDA(cudaMemcpyAsync(&nt, toff + N, sizeof(int64_t), cudaMemcpyDeviceToHost, s));
        KC_CUDA(cudaStreamSynchronize(s));
        *ntasks_out = nt;
    }
    int2* tasks;
    KC_TRY(A.get(&tasks, nt));
    ::kc::note_launch(), task_fill_k<<<blocks_for(N * 32, 256), 256, 0, s>>>(order, toff, N, tasks);
    KC_CUDA(cudaGetLastError());
    *tasks_out = tasks;
    if (count_out) *count_out = toff + N;
    return KC_OK;
}

// ---------------------------------------------------------------- launch core
// Everything one persistent launch needs.  kc_factor fills it with
// stream-ordered scratch; a kc_factor_plan keeps it across launches.
struct FactorCore {
    kc_pattern P;
    int prec = KC_FP32_FORM;
    int d = 2;
    const double* x = nullptr;
    int2* tasks = nullptr;
    const int64_t* ntasks = nullptr;  // device
    int maxr = 0;
    unsigned* done = nullptr;
    unsigned long long* ticket = nullptr;
    unsigned long long* zp = nullptr;
    int* status = nullptr;
    KernelParams kp{};
    const int32_t* col_set = nullptr;
    KernelParams* kps = nullptr;
    bool general = false;  // some set's kernel is not a closed-form Matern
    const double* aval = nullptr;  // given entries (kc_factor_given)
    int rpt = 128, lanes = 0, unroll = 8, warps = 8, hbits = 7, ctas = 0, adaptive = 0;
    int stage_req = 0;    // requested stage-buffer bytes of the bulk form: <= 0 ring or register form
    int stage_bytes = 0;  // chosen (0: ring or register form)
    int team = 1;         // warps that share one table
    int bulk_warps = 4;
    bool warps_auto = true;  // CTA size from the occupancy of the row tables
    long long spin = 4000000000LL;
    int hold = -1;
};

// The ring form: the default number of lanes per row, arrays on 16-byte boundaries.
static bool takes_ring(const FactorCore& F, const void* val) {
    const int lanes = F.prec == KC_FP64 ? RingLayout<double>::G : RingLayout<float>::G;
    const bool bulk = F.stage_bytes > 0 && !F.aval && !F.general;  // the other entry sources: ring or register form
    return !bulk && (F.lanes == 0 || F.lanes == lanes) && ((uintptr_t)F.P.col & 15) == 0 && ((uintptr_t)val & 15) == 0;
}

template <typename T, int U, int ENT>
static kc_status launch_core(const FactorCore& F, T* val, double* diag, cudaStream_t s) {
    FactorArgs<T> a;
    a.N = F.P.N;
    a.d = F.d;
    a.x = F.x;
    a.rowptr = F.P.rowptr;
    a.col = F.P.col;
    a.colptr = F.P.colptr;
    a.rowidx = F.P.rowidx;
    a.slot = F.P.slot;
    a.tasks = F.tasks;
    a.ntasks = F.ntasks;
    a.rpt = F.rpt;
    a.val = val;
    a.diag = diag;
    a.done = F.done;
    a.ticket = F.ticket;
    a.status = F.status;
    a.zero_piv = F.zp;
    a.kp = F.kp;
    a.aval = F.aval;
    a.col_set = F.col_set;
    a.kps = F.kps;
    a.spin_limit = F.spin;
    a.hold_col = F.hold;
    a.hbits = F.hbits;
    a.lanes = F.lanes;
    a.adaptive = F.adaptive;
    a.stage_bytes = F.stage_bytes;
    const bool bulk = ENT == 0 && F.stage_bytes > 0;
    const bool ring = takes_ring(F, val);
    const int team = bulk ? 1 : F.team;
    int dev = 0, optin = 0;
    KC_CUDA(cudaGetDevice(&dev));
    KC_CUDA(cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
    // one team's shared memory: the table, the control words, and per warp the ring (ring form) or two stage
    // buffers and two mbarriers (bulk form); 128-byte aligned
    auto layout = [&](int hbits) {
        a.hbits = hbits;
        a.ctl_off = (int)table_bytes<T>(hbits, team > 1);
        a.buf_off = a.ctl_off + (team > 1 ? 16 : 0);
        size_t b = a.buf_off;
        if (ring) b += (size_t)team * RING * RingLayout<T>::STAGE;
        if (bulk) b += 2 * (size_t)F.stage_bytes + 16;
        a.team_smem = (int)((b + 127) / 128 * 128);
    };
    layout(F.hbits);
    a.team = team;
    int warps = bulk ? F.bulk_warps : F.warps;
    if (bulk) {
        warps = std::min(warps, optin / a.team_smem);
        if (warps < 1) return fail(KC_EINVAL, "factor: stage_bytes too large for one warp's shared memory");
    } else if (!F.warps_auto) {  // a CTA size that was asked for: the largest table that fits it
        while (a.hbits > 7 && (size_t)(warps / team) * a.team_smem > (size_t)optin) layout(a.hbits - 1);
    }
    void (*kfn)(FactorArgs<T>) = nullptr;
    if constexpr (ENT == 0) {
        if (bulk) kfn = ichol_bulk_k<T, U, 0>;
    }
    if (ring) kfn = team > 1 ? ichol_ring_k<T, ENT, true> : ichol_ring_k<T, ENT, false>;
    else if (!bulk) kfn = team > 1 ? ichol_persistent_k<T, U, ENT, true> : ichol_persistent_k<T, U, ENT, false>;
    int per_sm = 0;
    KC_TRY(allow_dynamic_smem(kfn));
    if (!bulk && F.warps_auto) {
        // CTA size with the most resident warps (whole teams).  A smaller CTA must
        // win by over 20%: filling the shared memory to the last CTA leaves the
        // L1 cache too small.
        int best = 0;
        for (int w = 8; w >= team; w >>= 1) {
            const size_t sm_w = (size_t)(w / team) * a.team_smem;
            int n = 0;
            KC_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kfn, w * 32, sm_w));
            if (n * w * 5 > best * 6) {
                best = n * w;
                warps = w;
            }
        }
    }
    size_t smem = (size_t)(warps / team) * a.team_smem;
    KC_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kfn, warps * 32, smem));
    if (F.ctas > 0 && F.ctas < per_sm) per_sm = F.ctas;
    if (F.ctas < 0) per_sm = std::max(1, per_sm + F.ctas);  // leave -ctas CTA slots per SM to other streams
    if (per_sm < 1) return fail(KC_EINVAL, "factor: shared memory of one CTA exceeds the SM (stage_bytes too large?)");
    int64_t grid = (int64_t)sm_count() * per_sm;
    if (!bulk && F.ctas == 0 && F.warps_auto) {
        // Narrow levels (small sets): about one team per task of a level, the same
        // number on every SM.  The tasks go out in level order, so further teams
        // would only wait, and with several tasks on some SMs and none on others a
        // level takes as long as the fullest SM (2000 points, FP32 form: 1.73 ms
        // with every slot of the chip taken, 0.66 with 4 warps per SM; 100,003
        // points: 5.0 with 24 per SM, 4.0 with 16).
        const double want = 1.1 * team * (double)tasks_bound(&F.P, F.rpt) / (double)std::max(1, F.P.depth);
        while (warps > std::max(team, 4) && want < (double)warps * sm_count()) warps >>= 1;
        const int64_t ctas = std::max((int64_t)1, (int64_t)(want / ((double)warps * sm_count()) + 0.5));
        grid = std::min(grid, ctas * sm_count());
    }
    a.crowded = grid == (int64_t)sm_count() * per_sm;
    ::kc::note_launch(), done_init_k<<<blocks_for(F.P.N, 256), 256, 0, s>>>(F.P.colptr, F.P.rowptr, F.P.N, F.rpt,
                                                                           F.adaptive, team, F.done);
    KC_CUDA(cudaMemsetAsync(F.ticket, 0, sizeof(unsigned long long), s));
    KC_CUDA(cudaMemsetAsync(F.zp, 0, sizeof(unsigned long long), s));
    KC_CUDA(cudaMemsetAsync(F.status, 0, sizeof(int), s));
    smem = (size_t)(warps / team) * a.team_smem;
    ::kc::note_launch(), kfn<<<(unsigned)grid, warps * 32, smem, s>>>(a);
    KC_CUDA(cudaGetLastError());
    return KC_OK;
}

// The closed-form Matern kernels take the unroll asked for (register form); the
// other entry sources have one instantiation per precision (8 loads in flight per
// lane in the FP32 form, 4 in FP64).  All of them run in the ring form by default.
// The covariance functions behind calls (ENT = 1) spill 80 to 108 bytes there, what
// is kept across the calls; their calls take far longer (100,003 points, nu = 0.8,
// FP32 form: 6.3 ms beside 3.4 for nu = 5/2).
static kc_status launch_any(const FactorCore& F, void* val, double* diag, cudaStream_t s) {
    if (F.aval)
        return F.prec == KC_FP64 ? launch_core<double, 4, 2>(F, (double*)val, diag, s)
                                 : launch_core<float, 8, 2>(F, (float*)val, diag, s);
    if (F.general)
        return F.prec == KC_FP64 ? launch_core<double, 4, 1>(F, (double*)val, diag, s)
                                 : launch_core<float, 8, 1>(F, (float*)val, diag, s);
    if (F.prec == KC_FP64)
        return F.unroll >= 8 ? launch_core<double, 8, 0>(F, (double*)val, diag, s)
                             : launch_core<double, 4, 0>(F, (double*)val, diag, s);
    if (F.unroll >= 16) return launch_core<float, 16, 0>(F, (float*)val, diag, s);
    return F.unroll >= 8 ? launch_core<float, 8, 0>(F, (float*)val, diag, s)
                         : launch_core<float, 4, 0>(F, (float*)val, diag, s);
}

static kc_status read_status(const FactorCore& F, int64_t* zero_out, cudaStream_t s) {
    int h_status = 0;
    unsigned long long h_zp = 0;
    KC_CUDA(cudaMemcpyAsync(&h_status, F.status, sizeof(int), cudaMemcpyDeviceToHost, s));
    KC_CUDA(cudaMemcpyAsync(&h_zp, F.zp, sizeof(unsigned long long), cudaMemcpyDeviceToHost, s));
    KC_CUDA(cudaStreamSynchronize(s));
    if (zero_out) *zero_out = (int64_t)h_zp;
    if (h_status == DEV_TIMEOUT) return fail(KC_ETIMEOUT, "factor: a dependency wait ran out");
    if (h_status != 0) return fail(KC_ECUDA, "factor: device status " + std::to_string(h_status));
    return KC_OK;
}

static kc_status apply_opts(FactorCore& F, const kc_opts* o) {
    F.rpt = (o && o->rows_per_task > 0) ? o->rows_per_task : 0;  // 0: from the level width (auto_rows)
    F.warps = (o && o->warps_per_cta > 0) ? o->warps_per_cta : 8;
    F.warps_auto = !(o && o->warps_per_cta > 0);
    if (F.warps > 8) return fail(KC_EINVAL, "warps_per_cta must be <= 8");
    F.spin = (o && o->spin_limit_cycles > 0) ? o->spin_limit_cycles : 4000000000LL;
    F.ctas = o ? o->ctas_per_sm : 0;
    F.hold = (o && o->test_hold_column > 0) ? o->test_hold_column - 1 : -1;
    F.lanes = 0;
    if (o && o->lanes_per_row > 0) {
        int L = o->lanes_per_row;
        if (L > 32 || (L & (L - 1))) return fail(KC_EINVAL, "lanes_per_row must be a power of two <= 32");
        F.lanes = L;
    }
    F.unroll = (o && o->unroll > 0) ? o->unroll : 0;  // 0: from the mean row length (pick_hash)
    F.stage_req = o ? o->stage_bytes : 0;
    if (F.stage_req > 65536) return fail(KC_EINVAL, "stage_bytes must be <= 65536");
    F.adaptive = (o && o->adaptive_chunks) ? 1 : 0;
    if (F.unroll != 0 && F.unroll != 4 && F.unroll != 8 && F.unroll != 16)
        return fail(KC_EINVAL, "unroll must be 4, 8 or 16");
    return KC_OK;
}

static void pick_hash(FactorCore& F) {
    // table of the longest row, a power of two in 128..4096 slots; a longer row
    // falls back to binary search in global memory
    int hb = 7;
    while (hb < 12 && table_rows(hb) < F.maxr) ++hb;
    F.hbits = hb;
    // staging depth: 16 loads per lane in flight for long rows (FP32 form),
    // else 8; the FP64 form takes at most 8
    if (F.unroll == 0) F.unroll = F.prec == KC_FP64 ? 4 : (F.P.nnz >= 400 * F.P.N ? 16 : 8);
    // bulk form (on request): stage buffers of the requested size; a row
    // prefix longer than a buffer is merged from global memory
    F.stage_bytes = F.stage_req <= 0 ? 0 : std::max(64, (F.stage_req + 15) / 16 * 16);
    F.bulk_warps = F.warps < 4 ? F.warps : 4;
}

// Warps that share one table: so many that a warp's part of it is at most
// 6 KB (FP64: 6 KB of its 12 bytes per slot), which keeps 24 warps per SM
// beside their rings, as a divisor of the CTA's warps (CTAs of 3, 5 or 7 warps are
// teams as a whole: 131,071 points of the cube, rho = 4, FP64, 3 warps: 397 ms with a
// table a warp).  With the rows of a task asked for, no more than there are rounds of
// rows in it, for the others would only help to stage (40,000 points of the cube,
// rho = 4, FP32 form, 4 rows a task: 45 ms with a warp a task, 75 with teams of two).
static void pick_team(FactorCore& F) {
    const int round = F.prec == KC_FP64 ? RingLayout<double>::RR : RingLayout<float>::RR;
    const int most = F.rpt > 0 ? std::min(F.warps, std::max(1, F.rpt / round)) : F.warps;
    F.team = 1;
    for (int w = 1; w <= most && F.stage_bytes == 0; ++w)
        if (F.warps % w == 0) {
            F.team = w;
            if (((size_t)8 << F.hbits) <= (size_t)w * 6144) break;
        }
}

// Rows per task, unless set.  With R rows per level in the mean, a warp gets
// the larger of R / resident warps (24 per SM; in the FP64 form, with its
// larger tables and rings, 16), so that a level is about one task per warp,
// and, on narrow levels, R / (6 per SM) as long as these rows hold at most
// about 4500 entries: tasks shorter than that are mostly prologue (20,000
// points, FP32 form: 4 rows 2.4 ms, 16 rows 1.6; 100,003 points: 16 rows 4.3,
// 32 rows 4.0; 40,000 points of the cube, rho = 4: 8 rows 21.5, 16 rows 26.0).
// A power of two from one step of the ring form's rows to 128.
static void auto_rows(FactorCore& F) {
    if (F.rpt > 0) return;
    const bool f64 = F.prec == KC_FP64;
    const double sms = (double)sm_count(), nnz = (double)(F.P.nnz - F.P.N);
    const double level = nnz / (double)std::max(1, F.P.depth);
    const double narrow = std::min(level / (sms * 6.0), 4500.0 * (double)F.P.N / std::max(1.0, nnz));
    const double per = std::max(narrow, level / (sms * (f64 ? 16.0 : 24.0)));
    int r = f64 ? RingLayout<double>::RR : RingLayout<float>::RR;
    while (r < 128 && per > r * 1.41421356) r <<= 1;
    F.rpt = r * F.team;
}

// One factorisation: entries from the covariance function kern at the
// points x, or (kern NULL) the given matrix aval on the pattern.
static kc_status factor_run(const kc_pattern* P, const double* x, int d, const kc_kernel* kern, const double* aval,
                            int prec, void* val, double* diag, int64_t* zero_out, const kc_opts* o, cudaStream_t s) {
    if (prec != KC_FP64 && prec != KC_FP32_FORM) return fail(KC_EINVAL, "prec must be KC_FP64 or KC_FP32_FORM");
    FactorCore F;
    if (kern) {
        KC_TRY(kernel_params(kern, &F.kp));
        F.general = F.kp.nu_code > 2;
    } else {
        F.aval = aval;
    }
    KC_TRY(apply_opts(F, o));
    F.P = *P;
    F.prec = prec;
    F.d = d;
    F.x = x;
    Arena A(s);
    KC_TRY(upload_coef(F.kp, A, s));
    KC_TRY(max_row(P, A, s, &F.maxr));
    pick_hash(F);
    pick_team(F);
    auto_rows(F);
    KC_TRY(build_tasks(P, F.rpt, A, s, &F.tasks, &F.ntasks, nullptr, F.adaptive != 0));
    KC_TRY(A.get(&F.done, P->N));
    KC_TRY(A.get(&F.ticket, 1));
    KC_TRY(A.get(&F.zp, 1));
    KC_TRY(A.get(&F.status, 1));
    cudaEvent_t e0, e1;
    KC_CUDA(cudaEventCreate(&e0));
    KC_CUDA(cudaEventCreate(&e1));
    KC_CUDA(cudaEventRecord(e0, s));
    kc_status st = launch_any(F, val, diag, s);
    if (st != KC_OK) return st;
    KC_CUDA(cudaEventRecord(e1, s));
    st = read_status(F, zero_out, s);
    float ms = 0.f;
    if (cudaEventElapsedTime(&ms, e0, e1) == cudaSuccess) set_factor_kernel_ms(ms);
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    return st;
}

kc_status factor_impl(const kc_pattern* P, const double* x, int d, const kc_kernel* kern, int prec, void* val,
                      double* diag, int64_t* zero_out, const kc_opts* o, cudaStream_t s) {
    return factor_run(P, x, d, kern, nullptr, prec, val, diag, zero_out, o, s);
}

kc_status factor_given_impl(const kc_pattern* P, const double* aval, int prec, void* val, double* diag,
                            int64_t* zero_out, const kc_opts* o, cudaStream_t s) {
    return factor_run(P, nullptr, 0, nullptr, aval, prec, val, diag, zero_out, o, s);
}

}  // namespace kc

// ------------------------------------------------------------------ plans
// A plan keeps the task list and the counters of one pattern so that the
// factorisation is a single capturable launch (no allocation, no host sync).
struct kc_factor_plan {
    kc::FactorCore F;
    std::vector<void*> owned;
};

namespace kc {

static kc_status plan_alloc(kc_factor_plan* pl, void** p, size_t bytes) {
    cudaError_t e = cudaMalloc(p, bytes ? bytes : 16);
    if (e != cudaSuccess) return cuda_fail(e, "cudaMalloc(plan)");
    pl->owned.push_back(*p);
    return KC_OK;
}

kc_status plan_create_impl(const kc_pattern* P, const double* x, int d, const kc_kernel* kerns, int nsets,
                           const int32_t* col_set, int prec, const kc_opts* o, kc_factor_plan** out, cudaStream_t s) {
    if (prec != KC_FP64 && prec != KC_FP32_FORM) return fail(KC_EINVAL, "prec must be KC_FP64 or KC_FP32_FORM");
    if (nsets < 1 || (nsets > 1 && !col_set)) return fail(KC_EINVAL, "nsets >= 1; col_set required when nsets > 1");
    kc_factor_plan* pl = new kc_factor_plan();
    FactorCore& F = pl->F;
    auto bail = [&](kc_status st) {
        for (void* p : pl->owned) cudaFree(p);
        delete pl;
        return st;
    };
    kc_status st = kernel_params(&kerns[0], &F.kp);
    if (st == KC_OK) st = apply_opts(F, o);
    if (st != KC_OK) return bail(st);
    F.general = F.kp.nu_code > 2;
    F.P = *P;
    F.prec = prec;
    F.d = d;
    F.x = x;
    F.col_set = nsets > 1 ? col_set : nullptr;
    {
        Arena A(s);
        if ((st = max_row(P, A, s, &F.maxr)) != KC_OK) return bail(st);
        pick_hash(F);
        pick_team(F);
        auto_rows(F);
        int2* t;
        const int64_t* count;
        int64_t nt = 0;
        int64_t* kept;
        st = build_tasks(P, F.rpt, A, s, &t, &count, &nt, F.adaptive != 0);
        if (st != KC_OK) return bail(st);
        if ((st = plan_alloc(pl, (void**)&F.tasks, sizeof(int2) * nt)) != KC_OK) return bail(st);
        if ((st = plan_alloc(pl, (void**)&kept, 64)) != KC_OK) return bail(st);
        F.ntasks = kept;
        if (cudaMemcpyAsync(F.tasks, t, sizeof(int2) * nt, cudaMemcpyDeviceToDevice, s) != cudaSuccess ||
            cudaMemcpyAsync(kept, count, sizeof(int64_t), cudaMemcpyDeviceToDevice, s) != cudaSuccess)
            return bail(fail(KC_ECUDA, "plan: task copy"));
    }
    if ((st = plan_alloc(pl, (void**)&F.done, sizeof(unsigned) * P->N)) != KC_OK) return bail(st);
    if ((st = plan_alloc(pl, (void**)&F.ticket, 64)) != KC_OK) return bail(st);
    if ((st = plan_alloc(pl, (void**)&F.zp, 64)) != KC_OK) return bail(st);
    if ((st = plan_alloc(pl, (void**)&F.status, 64)) != KC_OK) return bail(st);
    if (F.kp.nu_code == 3) {
        double* tab;
        if ((st = plan_alloc(pl, (void**)&tab, sizeof(double) * KC_COEF_LEN)) != KC_OK) return bail(st);
        if ((st = upload_coef(F.kp, tab, s)) != KC_OK) return bail(st);
    }
    if (nsets > 1) {
        std::vector<KernelParams> h(nsets);
        for (int k = 0; k < nsets; ++k) {
            if ((st = kernel_params(&kerns[k], &h[k])) != KC_OK) return bail(st);
            if (h[k].nu_code > 2) F.general = true;
            if (h[k].nu_code == 3) {
                double* tab;
                if ((st = plan_alloc(pl, (void**)&tab, sizeof(double) * KC_COEF_LEN)) != KC_OK) return bail(st);
                if ((st = upload_coef(h[k], tab, s)) != KC_OK) return bail(st);
            }
        }
        if ((st = plan_alloc(pl, (void**)&F.kps, sizeof(KernelParams) * nsets)) != KC_OK) return bail(st);
        if (cudaMemcpy(F.kps, h.data(), sizeof(KernelParams) * nsets, cudaMemcpyHostToDevice) != cudaSuccess)
            return bail(fail(KC_ECUDA, "plan: kernel parameter copy"));
    }
    if (cudaStreamSynchronize(s) != cudaSuccess) return bail(fail(KC_ECUDA, "plan: synchronize"));
    *out = pl;
    return KC_OK;
}

kc_status plan_launch_impl(kc_factor_plan* pl, void* val, double* diag, cudaStream_t s) {
    return launch_any(pl->F, val, diag, s);
}

kc_status plan_finish_impl(kc_factor_plan* pl, int64_t* zero_out, cudaStream_t s) {
    return read_status(pl->F, zero_out, s);
}

// Pick lanes per row (the warp share of one row) and the staging depth by
// timing every combination once on the plan's own problem.  The ring form has
// no depth: its lanes are timed once, with the plan's depth.
kc_status plan_tune_impl(kc_factor_plan* pl, void* val, double* diag, int32_t* lanes_out, int32_t* unroll_out,
                         double* best_ms_out, cudaStream_t s) {
    FactorCore& F = pl->F;
    const int lanes_c[] = {2, 4, 8, 16};
    const int unroll_c[] = {8, 16};
    cudaEvent_t e0, e1;
    KC_CUDA(cudaEventCreate(&e0));
    KC_CUDA(cudaEventCreate(&e1));
    double best = 1e300;
    int bl = F.lanes, bu = F.unroll;
    const int depth = F.unroll;
    KC_TRY(launch_any(F, val, diag, s));  // warm-up
    KC_TRY(read_status(F, nullptr, s));
    for (int L : lanes_c)
        for (int U : unroll_c) {
            F.lanes = L;
            F.unroll = U;
            if (takes_ring(F, val)) {
                if (U != unroll_c[0]) continue;
                F.unroll = depth;
            }
            KC_CUDA(cudaEventRecord(e0, s));
            KC_TRY(launch_any(F, val, diag, s));
            KC_CUDA(cudaEventRecord(e1, s));
            KC_TRY(read_status(F, nullptr, s));
            float ms = 0.f;
            KC_CUDA(cudaEventElapsedTime(&ms, e0, e1));
            if (ms < best) {
                best = ms;
                bl = L;
                bu = F.unroll;
            }
        }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    F.lanes = bl;
    F.unroll = bu;
    if (lanes_out) *lanes_out = bl;
    if (unroll_out) *unroll_out = bu;
    if (best_ms_out) *best_ms_out = best;
    return KC_OK;
}

void plan_destroy_impl(kc_factor_plan* pl) {
    if (!pl) return;
    for (void* p : pl->owned) cudaFree(p);
    delete pl;
}

}  // namespace kc
