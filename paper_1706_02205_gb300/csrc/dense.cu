// The dense product Theta v of the refined solve for the closed-form Matern
// kernels, to the accuracy of FP64 sums with a fraction of their FP64 work.
//
// The FP64 pipe of the GB300 issues two lanes a clock and SM, so a product of
// N^2 entries, each a square root, an exponential and nrhs multiply-adds in
// FP64, took 30.6 ms at N = 16,384 with 16 right-hand sides, all of it that pipe.
// Here
//  - only the coordinate differences and the squared distance are FP64.  For
//    nu = 1/2 and 3/2 the rest of an entry is 64-bit integer arithmetic: the
//    square root by Newton steps from an FP32 seed, the exponential by a table of
//    2^(-j/256) and a short polynomial (P. T. P. Tang, ACM Trans. Math. Softw.
//    15 (1989) 144).  nu = 5/2 does the same in FP64 (19 operations);
//  - the multiply-adds go to the tensor cores by an error-free splitting
//    (K. Ozaki, T. Ogita, S. Oishi and S. M. Rump, Numer. Algorithms 59 (2012)
//    95): an entry Theta / sigma2 in [0, 1] is a 56-bit fixed-point number, eight
//    digits of 7 bits; a vector's 128 values under one power of two are 56-bit
//    numbers with sign, eight digits too; every product of digits and every sum
//    of 128 of them (up to eight pairs) is a whole number below 2^24, which the
//    FP16 products with FP32 sums of the tensor cores hold exactly.  Digit pairs
//    are summed by weight (a + b <= 8; what is left out is below 2^-60 of the
//    largest entry times the largest value), the nine sums of a block of 128 are
//    put together in 64-bit integers and added in FP64.
// A warp computes the entries of 16 rows and 16 columns at a time straight in
// the lanes that hold them as the first operand of mma.m16n8k16.
//
// N = 16,384: 4.1 ms with 16 right-hand sides (30.6 before), 3.3 ms with one
// (21.4); nu = 5/2: 11.7 ms; N = 40,000: 24.7 ms (194).  Against sums in 80-bit
// arithmetic the products of 777 to 1500 points are 1.1e-16 to 2.0e-16 off in
// the 2-norm, 1.0e-15 to 1.8e-15 before.  Bound by the integer multiplications
// and, from 16 right-hand sides on, by the 86 small products of 16 columns; two
// CTAs an SM instead of three (168 registers): 5.7 ms.  The check below, that no row
// loses by it, adds 0.06 ms to a product of 16 vectors.
#include <algorithm>
#include <cmath>

#include "dense.cuh"

namespace kc {

namespace {

constexpr int DT_WARPS = 4;             // warps per CTA
constexpr int DT_ROWS = 16 * DT_WARPS;  // rows per CTA
constexpr int DT_BLOCK = 128;           // columns per scale
constexpr int DIGITS = 8;
constexpr int LEVELS = 9;  // a + b = 0 .. 8
constexpr double R256_LN2 = 369.3299304675746;            // 256 / ln 2
constexpr double LN2_256_HI = 0.0027076061737716373;      // ln 2 / 256, its first 33 bits
constexpr double LN2_256_LO = 2.9064910585985925e-13;     // the rest
constexpr double TO_INT = 6755399441055744.0;             // 1.5 2^52: adding it rounds to a whole number

struct DenseArgs {
    const double* __restrict__ x;
    int64_t N;
    int d;
    int nu_code;
    double scale;
    const uint2* __restrict__ vf;     // digits of v as second operands
    const double* __restrict__ coef;  // [block][16]: sigma2 2^(e - 42)
    const double* __restrict__ tab;   // 2^(-j/256)
    const unsigned long long* __restrict__ itab;  // 2^63 times that
    unsigned long long smant;         // scale = smant 2^sexp, smant in [2^63, 2^64)
    int sexp;
    int64_t blocks_per_split;
    int ns;
    double* out;  // [split][N][ns]
    const int* exact;  // nonzero: leave this product to FP64
};

__device__ __forceinline__ uint32_t half2_sub(uint32_t a, uint32_t b) {
    uint32_t r;
    asm("sub.rn.f16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
    return r;
}
// two digits (0..128) as a pair of FP16 numbers: 1024 + d has the bits 0x6400 | d
__device__ __forceinline__ uint32_t digit_pair(uint32_t lo, uint32_t hi) {
    return half2_sub((lo | (hi << 16)) | 0x64006400u, 0x64006400u);
}
__device__ __forceinline__ void mma_16816(float (&c)[4], const uint32_t (&a)[4], uint2 b) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b.x), "r"(b.y));
}

// Theta / sigma2 at squared distance s as a multiple of 2^-56, rounded to nearest.
__device__ __forceinline__ unsigned long long entry_fixed(double s, int nu_code, double scale, const double* tab) {
    const int hi = __double2hiint(s), lo = __double2loint(s);
    const int ex = (hi >> 20) - 1023;
    double r;
    if (ex <= -1022 || ex >= 1024) {
        r = sqrt(s);  // zero, denormal, infinite
    } else {
        // s = m 4^q, 1 <= m < 4; the root of m by two Newton steps g += (m - g^2) / (2 sqrt(m))
        const int par = ex & 1, top = hi & 0xfffff;
        const double m = __hiloint2double(top | ((1023 + par) << 20), lo);
        const unsigned yb =
            __float_as_uint(rsqrtf(__uint_as_float(((127 + par) << 23) | (top << 3) | ((unsigned)lo >> 29))));
        const int yh = (int)(yb >> 3) + (896 << 20), yl = (int)(yb << 29);
        const double y = __hiloint2double(yh, yl), h = __hiloint2double(yh - (1 << 20), yl);
        double g = m * y;
        g = fma(fma(-g, g, m), h, g);
        g = fma(fma(-g, g, m), h, g);
        r = __hiloint2double(__double2hiint(g) + (((ex - par) >> 1) << 20), __double2loint(g));
    }
    const double t = r * scale;
    if (!(t < 50.0)) return 0ull;  // (1 + t + t^2 / 3) e^-t < 2^-62
    // e^-t = 2^(-n / 256) e^-f, |f| <= ln 2 / 512
    const double z = fma(t, R256_LN2, TO_INT);
    const int n = __double2loint(z);
    const double nd = z - TO_INT;
    double f = fma(nd, -LN2_256_HI, t);
    f = fma(nd, -LN2_256_LO, f);
    double a = fma(f, 1.0 / 24.0, -1.0 / 6.0);
    a = fma(f, a, 0.5);
    a = fma(f, a, -1.0);
    const double tj = tab[n & 255];
    double v = fma(tj, f * a, tj);
    if (nu_code == 1) v *= 1.0 + t;
    else if (nu_code == 2) v *= fma(t * (1.0 / 3.0), t, 1.0 + t);
    const int vh = __double2hiint(v);
    const int sh = (n >> 8) - ((vh >> 20) - 1023) - 4;  // v 2^-(n>>8) 2^56 = mantissa >> sh
    const unsigned long long man =
        ((unsigned long long)((vh & 0xfffff) | (1 << 20)) << 32) | (unsigned)__double2loint(v);
    if (sh <= 0) return man << -sh;
    if (sh > 60) return 0ull;
    return (man + (1ull << (sh - 1))) >> sh;
}

// The same in 64-bit integers, for nu = 1/2 and 3/2: the FP64 pipe issues one
// operation in the time of 16 integer instructions of the four schedulers.
// Every fixed-point number below keeps at least 2^-56 of an entry's unit.
__device__ __forceinline__ unsigned long long entry_fixed_int(double s, int nu_code, const DenseArgs& A,
                                                              const double* tab, const unsigned long long* itab) {
    const int hi = __double2hiint(s);
    const unsigned lo = (unsigned)__double2loint(s);
    const int ex = (hi >> 20) - 1023;
    if (ex <= -1022 || ex >= 1024) return s == 0.0 ? 1ull << 56 : entry_fixed(s, nu_code, A.scale, tab);
    // s = m 4^q, 1 <= m < 4, M = m 2^62; g = sqrt(m), G = g 2^62, by two Newton steps
    // g += (m - g^2) y / 2 with y an FP32 approximation of 1 / sqrt(m)
    const int par = ex & 1, top = hi & 0xfffff;
    const unsigned long long M = (((unsigned long long)(unsigned)(top | 0x100000) << 32) | lo) << (10 + par);
    const float y = rsqrtf(__uint_as_float(((127 + par) << 23) | (top << 3) | (lo >> 29)));
    const unsigned Y = __float2uint_rz(y * 2147483648.0f);  // y 2^31
    const int Yh = (int)(Y >> 1);
    unsigned long long G = ((unsigned long long)(unsigned)(M >> 32) * Y << 1) + ((unsigned long long)(unsigned)M * Y >> 31);
    const long long e1 = (long long)((M >> 2) - __umul64hi(G, G));  // (m - g^2) 2^60, below 2^41
    G += (unsigned long long)(((long long)(int)(e1 >> 10) * Yh) >> 19);
    const long long e2 = (long long)((M >> 2) - __umul64hi(G, G));  // below 2^20
    G += (unsigned long long)(((long long)(int)e2 * Yh) >> 29);
    // t = r scale, T = t 2^57
    const int k = ((ex - par) >> 1) + A.sexp + 59;
    const unsigned long long H = __umul64hi(G, A.smant);
    if (k > 1) return 0ull;  // t >= 64
    const unsigned long long T = k >= 0 ? H << k : k > -64 ? H >> -k : 0ull;
    if (T >= 50ull << 57) return 0ull;
    // w = t 256 / ln 2 with 48 bits after the point: e^-t = 2^(-n / 256) e^-x, x = F / 256, F = frac(w) ln 2
    const unsigned long long W = __umul64hi(T, 0xb8aa3b295c17f0bcull);
    const int n = (int)(W >> 48);
    const unsigned long long F = __umul64hi(W << 16, 0xb17217f7d1cf79acull), F2 = __umul64hi(F, F);
    const unsigned f = (unsigned)(F >> 32), f2 = (unsigned)(F2 >> 32), f3 = __umulhi(f2, f);
    // 1 - e^-x = x - x^2/2 + x^3 (1/6 - x/24 + x^2/120)
    const unsigned c3 = 715827882u - __umulhi(f, 699050u) + __umulhi(f2, 546u);
    const unsigned long long D = (F >> 8) - (F2 >> 17) + ((unsigned long long)__umulhi(f3, c3) << 8);
    const unsigned long long tj = itab[n & 255];
    unsigned long long P = tj - __umul64hi(tj, D);  // e^-t 2^(63 + n / 256)
    int sh = n >> 8;
    if (nu_code == 1) P = __umul64hi(P, T + (1ull << 57));  // (1 + t) e^-t 2^56
    else sh += 7;
    if (sh == 0) return P;
    if (sh > 63) return 0ull;
    return (P + (1ull << (sh - 1))) >> sh;
}

// D: coordinates (0: any, from A.d); NT: groups of 8 right-hand sides
template <int D, int NT, bool INT>
__global__ void __launch_bounds__(32 * DT_WARPS, 3) dense_theta_mma_k(DenseArgs A) {
    __shared__ double tab[256];
    __shared__ unsigned long long itab[INT ? 256 : 1];
    if (*A.exact) return;
    for (int q = threadIdx.x; q < 256; q += 32 * DT_WARPS) {
        tab[q] = A.tab[q];
        if constexpr (INT) itab[q] = A.itab[q];
    }
    __syncthreads();
    const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    const int64_t j0 = (int64_t)blockIdx.x * DT_ROWS + (threadIdx.x >> 5) * 16 + g;  // the lane's rows: j0, j0 + 8
    const int64_t jr[2] = {min(j0, A.N - 1), min(j0 + 8, A.N - 1)};
    double xj[2][D > 0 ? D : 1];
    if constexpr (D > 0)
#pragma unroll
        for (int q = 0; q < 2; ++q)
#pragma unroll
            for (int c = 0; c < D; ++c) xj[q][c] = A.x[jr[q] * D + c];
    double y[NT][4] = {};
    const int64_t nblocks = (A.N + DT_BLOCK - 1) / DT_BLOCK;
    const int64_t b0 = (int64_t)blockIdx.y * A.blocks_per_split, b1 = min(nblocks, b0 + A.blocks_per_split);
    for (int64_t b = b0; b < b1; ++b) {
        float acc[NT][LEVELS][4] = {};
#pragma unroll 1
        for (int ks = 0; ks < DT_BLOCK / 16; ++ks) {
            const int64_t kb = b * DT_BLOCK + ks * 16;
            if (kb >= A.N) break;
            unsigned long long q[2][4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int64_t k = min(kb + 2 * t + (e & 1) + 8 * (e >> 1), A.N - 1);  // past the end: digits of v are 0
#pragma unroll
                for (int w = 0; w < 2; ++w) {
                    double s = 0.0;
                    if constexpr (D > 0) {
#pragma unroll
                        for (int c = 0; c < D; ++c) {
                            const double u = xj[w][c] - __ldg(&A.x[k * D + c]);
                            s = c == 0 ? u * u : fma(u, u, s);
                        }
                    } else {
                        for (int c = 0; c < A.d; ++c) {
                            const double u = __ldg(&A.x[jr[w] * A.d + c]) - __ldg(&A.x[k * A.d + c]);
                            s = fma(u, u, s);
                        }
                    }
                    if constexpr (INT) q[w][e] = entry_fixed_int(s, A.nu_code, A, tab, itab);
                    else q[w][e] = entry_fixed(s, A.nu_code, A.scale, tab);
                }
            }
            // first operand, digit by digit: rows g and g + 8, columns 2t, 2t + 1 and 8 further
            uint32_t af[DIGITS][4];
#pragma unroll
            for (int p = 0; p < 4; ++p) {
                const unsigned long long q0 = q[p & 1][(p >> 1) * 2], q1 = q[p & 1][(p >> 1) * 2 + 1];
                const uint32_t h0 = (uint32_t)(q0 >> 28), h1 = (uint32_t)(q1 >> 28);
                const uint32_t l0 = (uint32_t)q0 & 0xfffffffu, l1 = (uint32_t)q1 & 0xfffffffu;
                af[0][p] = digit_pair(h0 >> 21, h1 >> 21);
#pragma unroll
                for (int a = 1; a < 4; ++a)
                    af[a][p] = digit_pair((h0 >> (21 - 7 * a)) & 127u, (h1 >> (21 - 7 * a)) & 127u);
#pragma unroll
                for (int a = 0; a < 4; ++a)
                    af[4 + a][p] = digit_pair((l0 >> (21 - 7 * a)) & 127u, (l1 >> (21 - 7 * a)) & 127u);
            }
#pragma unroll
            for (int nt = 0; nt < NT; ++nt) {
                const uint2* bp = A.vf + (((b * (DT_BLOCK / 16) + ks) * NT + nt) * DIGITS) * 32 + lane;
#pragma unroll
                for (int c = 0; c < DIGITS; ++c) {
                    const uint2 bf = __ldg(bp + c * 32);
#pragma unroll
                    for (int a = 0; a < DIGITS; ++a)
                        if (a + c < LEVELS) mma_16816(acc[nt][a + c], af[a], bf);
                }
            }
        }
        // the block's nine sums of weight 2^(-14 - 7 s), whole numbers: exactly together, then into FP64
#pragma unroll
        for (int nt = 0; nt < NT; ++nt)
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                long long i1 = 0, i2 = 0;
#pragma unroll
                for (int s = 0; s < 5; ++s) i1 = i1 * 128 + __float2int_rn(acc[nt][s][i]);
#pragma unroll
                for (int s = 5; s < LEVELS; ++s) i2 = i2 * 128 + __float2int_rn(acc[nt][s][i]);
                const double c = __ldg(&A.coef[b * 16 + nt * 8 + 2 * t + (i & 1)]);
                y[nt][i] = fma(fma((double)i2, 1.0 / 268435456.0, (double)i1), c, y[nt][i]);
            }
    }
#pragma unroll
    for (int nt = 0; nt < NT; ++nt)
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int64_t j = j0 + (i >> 1) * 8;
            const int r = nt * 8 + 2 * t + (i & 1);
            if (j < A.N && r < A.ns) A.out[((int64_t)blockIdx.y * A.N + j) * A.ns + r] = y[nt][i];
        }
}

// v[k][r] (stride ns) by blocks of 128 columns: a power of two above the
// block's values, and their digits as second operands of the products (lane g 4
// + t: column g of the group, rows 2t, 2t + 1 and 8 further).  A block with a
// value that is not finite gets a NaN for a scale.
template <int NT>
__global__ void __launch_bounds__(128) dense_split_k(const double* __restrict__ v, int64_t N, int ns, double sigma2,
                                                     uint32_t* __restrict__ vf, double* __restrict__ coef,
                                                     double* __restrict__ bmax, const double* __restrict__ scale,
                                                     float* __restrict__ w, int* __restrict__ exact) {
    if (blockIdx.x == 0 && threadIdx.x == 0) *exact = 0;
    const int lane = threadIdx.x & 31;
    const int64_t b = blockIdx.x;
    for (int r = threadIdx.x >> 5; r < 8 * NT; r += 4) {
        double x[4];
        double mx = 0.0;
        bool fine = true;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int64_t k = b * DT_BLOCK + 4 * lane + i;
            x[i] = r < ns && k < N ? v[k * ns + r] : 0.0;
            if (r < ns && k < N) w[k * ns + r] = (float)(fabs(x[i]) * scale[r]);
            fine &= isfinite(x[i]) != 0;
            mx = fmax(mx, fabs(x[i]));
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        fine = __all_sync(0xffffffffu, fine);
        int e = 0;
        frexp(mx, &e);  // mx < 2^e
        const bool zero = !fine || mx == 0.0;
        unsigned long long mag[4];
        uint32_t sign[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            mag[i] = zero ? 0ull : (unsigned long long)__double2ll_rn(scalbn(fabs(x[i]), 56 - e));
            sign[i] = x[i] < 0.0 ? 0x8000u : 0u;
        }
        if (lane == 0) {
            const double c = zero ? 0.0 : scalbn(sigma2, e - 42);
            coef[b * 16 + r] = fine ? c : nan("");
            bmax[b * 16 + r] = fine ? mx : nan("");
        }
#pragma unroll
        for (int p = 0; p < 2; ++p) {
            const int k = 4 * lane + 2 * p, ks = k >> 4, kk = k & 15;
            uint32_t* dst = vf + ((((b * (DT_BLOCK / 16) + ks) * NT + (r >> 3)) * DIGITS) * 32 + (r & 7) * 4 +
                                  ((kk & 7) >> 1)) * 2 + (kk >> 3);
#pragma unroll
            for (int c = 0; c < DIGITS; ++c) {
                const uint32_t d0 = (uint32_t)(mag[2 * p] >> (49 - 7 * c)) & (c ? 127u : 255u);
                const uint32_t d1 = (uint32_t)(mag[2 * p + 1] >> (49 - 7 * c)) & (c ? 127u : 255u);
                dst[(int64_t)c * 64] = digit_pair(d0, d1) ^ (sign[2 * p] | (sign[2 * p + 1] << 16));
            }
        }
    }
}

// y = sum over the splits in order + nugget v
__global__ void dense_sum_k(const double* __restrict__ part, int splits, int64_t n, double nugget,
                            const double* __restrict__ v, double* __restrict__ y, const int* __restrict__ exact) {
    const int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= n || *exact) return;
    double s = part[q];
    for (int p = 1; p < splits; ++p) s += part[(int64_t)p * n + q];
    y[q] = fma(nugget, v[q], s);
}

// ---- Is every row as accurate as FP64 sums would make it?
// The split rounds entries to 2^-57 and a block's values to 2^-57 of its largest, so
// row j is off by some 2^-57 S, S the mean over the vector of its blocks' largest
// values, whatever the row's own weight T_j = sum_k Theta_jk |v_k| / sigma2 is.  FP64
// entries and sums are off by 5 to 20 units of 2^-53 T_j in a set's worst row.  Measured against
// 80-bit sums over 1000 points in two and three dimensions, three kernels, ranges of
// 0.05 to 0.3, random vectors and their solutions: the split's worst row and its rows
// of least weight are more accurate wherever T_j >= S / 17, and not all at S / 40;
// points far from all that is large (one-hot vectors, far clusters of other scales)
// lie far below.  T_j is estimated by L L^T |v| with the preconditioner's factor in floats
// (2 x nnz products beside the N^2; in doubles they took three times as long, 0.17 ms
// for 1.7 M entries and 16 vectors); a product with a row below S / 16 is left to FP64, as are
// values or points that are not finite.
constexpr double LEAST_WEIGHT = 1.0 / 16.0;

// scale = the power of two by which a vector like the right-hand side, over sigma2, is of size 1
__global__ void dense_scale_k(const double* __restrict__ norm2, int64_t N, double sigma2, int ns,
                              double* __restrict__ scale) {
    const int r = threadIdx.x;
    if (r >= 16) return;
    const double m = r < ns ? sqrt(norm2[r] / (double)N) : 0.0;
    scale[r] = m > 0.0 && m < INFINITY ? scalbn(1.0, max(-1000, min(1000, -ilogb(m) - ilogb(sigma2)))) : 1.0;
}

// Every block of 64 rows adds up S for itself, from 16 x nblocks values.
constexpr int CHECK_ROWS = 64;
__global__ void __launch_bounds__(256) dense_check_k(const double* __restrict__ bmax, const double* __restrict__ scale,
                                                     const float* __restrict__ tw, double sigma2,
                                                     const double* __restrict__ x, int64_t N, int64_t nblocks, int d,
                                                     int ns, int* __restrict__ exact) {
    __shared__ double sum[16][17];
    __shared__ float least[16];
    const int r = threadIdx.x & 15, g = threadIdx.x >> 4;
    double s = 0.0;
    if (r < ns)
        for (int64_t b = g; b < nblocks; b += 16) s += bmax[b * 16 + r] * (double)min((int64_t)DT_BLOCK, N - b * DT_BLOCK);
    sum[g][r] = s;
    __syncthreads();
    if (threadIdx.x < 16) {
        double t = 0.0;
        for (int q = 0; q < 16; ++q) t += sum[q][threadIdx.x];
        least[threadIdx.x] = (float)(LEAST_WEIGHT * sigma2 * (t / (double)N) * scale[threadIdx.x]);
    }
    __syncthreads();
    const int64_t n = N * ns, q0 = (int64_t)blockIdx.x * CHECK_ROWS * ns;
    bool bad = false;
    for (int64_t q = q0 + threadIdx.x; q < min(n, q0 + CHECK_ROWS * ns); q += 256) {
        const int c = (int)(q & (ns - 1));
        bad |= !(tw[q] >= least[c]) || !(tw[q] < INFINITY);
        if (c == 0)
            for (int t = 0; t < d; ++t) bad |= !isfinite(x[q / ns * d + t]);
    }
    if (bad) *exact = 1;
}

template <int NT>
kc_status launch(const DenseSplit& S, DenseArgs a, const double* v, double sigma2, double nugget, double* y,
                 cudaStream_t s) {
    const int64_t nblocks = (a.N + DT_BLOCK - 1) / DT_BLOCK;
    ::kc::note_launch(), dense_split_k<NT><<<(unsigned)nblocks, 128, 0, s>>>(v, a.N, a.ns, sigma2, (uint32_t*)S.vf,
                                                                          S.coef, S.bmax, S.scale, S.w, S.exact);
    KC_CUDA(cudaGetLastError());
    KC_TRY(S.LL.apply(S.w, S.tw, s));
    ::kc::note_launch(), dense_check_k<<<blocks_for(a.N, CHECK_ROWS), 256, 0, s>>>(S.bmax, S.scale, S.tw, sigma2, a.x, a.N,
                                                                                  nblocks, a.d, a.ns, S.exact);
    const int64_t n = a.N * a.ns;
    const dim3 grid(blocks_for(a.N, DT_ROWS), (unsigned)S.splits);
    void (*kfn)(DenseArgs);
    if (a.nu_code < 2)
        kfn = a.d == 1   ? dense_theta_mma_k<1, NT, true>
              : a.d == 2 ? dense_theta_mma_k<2, NT, true>
              : a.d == 3 ? dense_theta_mma_k<3, NT, true>
                         : dense_theta_mma_k<0, NT, true>;
    else
        kfn = a.d == 1   ? dense_theta_mma_k<1, NT, false>
              : a.d == 2 ? dense_theta_mma_k<2, NT, false>
              : a.d == 3 ? dense_theta_mma_k<3, NT, false>
                         : dense_theta_mma_k<0, NT, false>;
    ::kc::note_launch(), kfn<<<grid, 32 * DT_WARPS, 0, s>>>(a);
    ::kc::note_launch(), dense_sum_k<<<blocks_for(n, 256), 256, 0, s>>>(S.part, S.splits, n, nugget, v, y, S.exact);
    KC_CUDA(cudaGetLastError());
    return KC_OK;
}

}  // namespace

kc_status dense_split_init(DenseSplit& S, const kc_pattern* P, int prec, const void* val, const double* diag,
                           double sigma2, const double* norm2, int ns, Arena& A, cudaStream_t s) {
    const int64_t N = P->N;
    const int64_t nblocks = (N + DT_BLOCK - 1) / DT_BLOCK, rows = (N + DT_ROWS - 1) / DT_ROWS;
    // column ranges so that there are about 16 CTAs per SM (three are resident: the last wave is then
    // a small part), at most 32, each of whole blocks
    const int64_t want = std::min<int64_t>(32, (16 * (int64_t)sm_count() + rows - 1) / rows);
    S.per = (nblocks + want - 1) / std::max<int64_t>(1, want);
    S.splits = (int)((nblocks + S.per - 1) / S.per);
    S.nt = ns > 8 ? 2 : 1;
    KC_TRY(A.get(&S.vf, nblocks * (DT_BLOCK / 16) * S.nt * DIGITS * 32));
    KC_TRY(A.get(&S.coef, nblocks * 16));
    KC_TRY(A.get(&S.part, (int64_t)S.splits * N * ns));
    KC_TRY(A.get(&S.tab, 512));
    KC_TRY(A.get(&S.bmax, nblocks * 16));
    KC_TRY(A.get(&S.w, N * ns));
    KC_TRY(A.get(&S.tw, N * ns));
    KC_TRY(A.get(&S.exact, 1));
    KC_TRY(A.get(&S.scale, 16));
    ::kc::note_launch(), dense_scale_k<<<1, 32, 0, s>>>(norm2, N, sigma2, ns, S.scale);
    KC_TRY(S.LL.init(P, prec, val, diag, ns, A, s));
    // 2^(-j/256) as doubles and as whole multiples of 2^-63: the 64-bit mantissas by eight
    // square roots of 1/2 multiplied up in integers (the host's long double is a double on some machines)
    double h[512];
    unsigned long long* u = (unsigned long long*)(h + 256);
    unsigned __int128 root[8];  // 2^(-2^-(b+1)) 2^64, b = 0 .. 7
    for (int b = 0; b < 8; ++b) {
        const unsigned __int128 of = b == 0 ? (unsigned __int128)1 << 63 : root[b - 1];  // its square, 2^64 units
        unsigned __int128 lo = 0, hi = ((unsigned __int128)1 << 64) - 1;
        while (lo < hi) {  // largest r with r^2 <= of 2^64
            const unsigned __int128 mid = (lo + hi + 1) >> 1;
            if (mid * mid <= of << 64) lo = mid;
            else hi = mid - 1;
        }
        root[b] = lo;
    }
    for (int j = 0; j < 256; ++j) {
        unsigned __int128 v = (unsigned __int128)1 << 64;
        for (int b = 0; b < 8; ++b)
            if ((j >> (7 - b)) & 1) v = (v * root[b] + ((unsigned __int128)1 << 63)) >> 64;
        h[j] = exp2(-j / 256.0);
        u[j] = (unsigned long long)(v >> 1);
    }
    KC_CUDA(cudaMemcpyAsync(S.tab, h, sizeof(h), cudaMemcpyHostToDevice, s));  // pageable: copied before it returns
    return KC_OK;
}

kc_status dense_theta_split(const DenseSplit& S, const double* x, int64_t N, int d, const KernelParams& kp,
                            const double* v, double* y, int ns, cudaStream_t s) {
    DenseArgs a;
    a.x = x;
    a.N = N;
    a.d = d;
    a.nu_code = kp.nu_code;
    a.scale = kp.scale;
    a.vf = S.vf;
    a.coef = S.coef;
    a.tab = S.tab;
    a.itab = (const unsigned long long*)(S.tab + 256);
    int e = 0;
    const double m = frexp(kp.scale, &e);  // scale = m 2^e, 1/2 <= m < 1
    a.smant = (unsigned long long)(m * 18446744073709551616.0);
    a.sexp = e - 64;
    a.blocks_per_split = S.per;
    a.ns = ns;
    a.out = S.part;
    a.exact = S.exact;
    return S.nt == 2 ? launch<2>(S, a, v, kp.sigma2, kp.nugget, y, s) : launch<1>(S, a, v, kp.sigma2, kp.nugget, y, s);
}

}  // namespace kc
