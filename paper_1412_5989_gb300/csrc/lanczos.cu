// Lanczos for the lowest eigenpairs (Sec. 2: successive matrix-vector
// products and orthogonalisations), for K matrices that share one half-stored
// structure, all K Krylov sequences advancing together.
//
// Device:
//   - y = H x reads each stored nonzero of the upper half once: the row part
//     as double-float sums of FP32-pair products, the mirrored half added to
//     64-bit fixed-point column accumulators (integer atomic adds commute, so
//     y is deterministic); no FP64 operation per nonzero;
//   - over row shards held by several processes, each multiplies its own rows
//     and a caller callback sums the two product buffers across them;
//   - values element-major (the K values of a nonzero together) and vectors
//     element-major x[i * K + s], FP64;
//   - full reorthogonalisation: classical Gram-Schmidt applied twice, dot
//     products reduced in two fixed-order stages;
//   - one step ahead of the host: the scalars of a step reach it while the next
//     step runs.
// Host: per set (sets on parallel host threads), the residual bound of the
// nev-th pair from a Sturm bisection and a twisted factorisation of the
// tridiagonal, O(m) a step; once that pair is near its bound, the lowest Ritz values
// and all residual bounds beta_m |z_m| from implicit-QR sweeps that rotate only
// the last row of the eigenvector matrix; the lowest Ritz vector's coefficients by
// inverse iteration.
// One GB300, whole solves: 800 rows 4.2 ms; 143,792 rows with set-up and gradient 37
// ms; 64 sets of 48,917 rows 325 ms; the uneven batch of 197,822 / 143,792 / 814,092
// rows 394 ms.
#include <algorithm>
#include <cmath>
#include <mutex>
#include <thread>
#include <vector>

#include "cih_internal.h"
#include "ham_common.cuh"

namespace cih {
namespace {

// fn(s) for s = 0 .. K - 1, on up to 8 host threads when there is more than one set
template <class F>
void parallel_sets(int K, F &&fn)
{
    const int nt = std::min({K, 8, (int)std::max(1u, std::thread::hardware_concurrency())});
    if (nt <= 1) {
        for (int s = 0; s < K; ++s) fn(s);
        return;
    }
    std::vector<std::thread> th;
    for (int t = 0; t < nt; ++t)
        th.emplace_back([&, t]() {
            for (int s = t; s < K; s += nt) fn(s);
        });
    for (auto &x : th) x.join();
}

constexpr int kSumsqBlocks = 256;                // partial sums of the bound
constexpr int kDotBlocks = 256;
constexpr int kThreads = 256;

// element-major values: vem[k * K + s] = val[s * nnz + k]
__global__ void k_vals_em(int K, int64_t nnz, const float *val, float *vem)
{
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < nnz * K; t += (int64_t)gridDim.x * blockDim.x) {
        const int64_t k = t / K;
        const int s = (int)(t - k * K);
        vem[t] = val[(int64_t)s * nnz + k];
    }
}

// Rows [r0, r1) of the matrix whose column and value arrays start at stored
// nonzero `base` (0 for a whole matrix; rowptr[r0] for a row shard).
struct RowRange {
    int64_t r0, r1, base;
};

// ---- y = H x from the stored upper half, each stored nonzero read once.
//
// Row i's warp forms the row part sum_j h_ij x_j (double-float sums in a
// fixed order: lanes, then a shuffle tree), and sends each strictly-upper h_ij x_i
// to column j's accumulator as a 64-bit fixed-point integer (units 2^-s) by
// an atomic add.  Integer adds commute, so y does not depend on the order in
// which rows run: the product is deterministic without a transposed copy.
// k_sym_finish adds the two parts and clears the accumulators.
//
// The scale 2^s keeps every accumulator inside 2^60: for column j,
// |sum_{i<j} h_ij x_i| <= ||h_{.j}|| ||x|| (Cauchy-Schwarz) <= F ||x||, with
// F the Frobenius norm of the strictly-upper part over all sets, and the
// Lanczos vectors have ||x|| = 1.  Each product, an FP32 pair, enters as its
// rounded hi plus its rounded lo: at most one unit 2^-s of absolute error.

// partial[blk] = this block's sum of the squares of the strictly-upper values of
// all sets, in double-float sums of the exact FP32-pair squares.  A warp takes R
// rows at a time and streams their values, whatever row they are of, 512 at a
// time: four float4 a lane, the next four in flight while these are summed; the K
// values of a row's first element, the diagonal, are set to zero where they fall
// into the stretch.  Bound by HBM and the latency at each change of rows.  A loop
// over each row with one float a lane and load took, at 4+4 Nmax=6, 0.93 ms
// (4.0 TB/s) against 0.82 ms, and at 64 sets of 3+4 Nmax=4 0.68 against 0.41 ms; runs of
// equal length for all warps, found by a search, 0.23 ms there but 1.11 ms for one set.
// R = 8 / K rows (at least one): 4 to 16 for one set are alike, 31 leave warps idle.
// Blocks beyond gridDim.x have no part: their partials are zero.
constexpr int kSumsqThreads = 1024, kSumsqGrid = 152;              // one block on each of GB300's SMs, 32 warps
__global__ void __launch_bounds__(kSumsqThreads) k_upper_sumsq(RowRange rr, int K, const int64_t *rowptr,
                                                               const float *vem, double *partial)
{
    __shared__ double red[kSumsqThreads / 32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int64_t nw = (int64_t)gridDim.x * (kSumsqThreads / 32), w = blockIdx.x * (int64_t)(kSumsqThreads / 32) + wid;
    const int64_t skip = ((uintptr_t)vem >> 2) & 3;                // floats by which vem is past a 16-byte boundary
    const int R = max(1, 8 / K);
    DF acc[4] = {df_of(0.f), df_of(0.f), df_of(0.f), df_of(0.f)};
    for (int64_t i0 = rr.r0 + w * R; i0 < rr.r1; i0 += nw * R) {
        const int64_t win = (rowptr[min(i0 + min(lane, R), rr.r1)] - rr.base) * K;      // row starts; lane R: the end
        const int64_t lo = __shfl_sync(0xffffffffu, win, 0), hi = __shfl_sync(0xffffffffu, win, R);
        auto load = [&](int64_t b, float4 (&x)[4]) {
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int64_t t = b + 128 * q + 4 * lane;
                if (t >= lo && t + 4 <= hi) {
                    x[q] = __ldcs(reinterpret_cast<const float4 *>(vem + t));
                } else {
                    x[q].x = t >= lo && t < hi ? vem[t] : 0.f;
                    x[q].y = t + 1 >= lo && t + 1 < hi ? vem[t + 1] : 0.f;
                    x[q].z = t + 2 >= lo && t + 2 < hi ? vem[t + 2] : 0.f;
                    x[q].w = t + 3 >= lo && t + 3 < hi ? vem[t + 3] : 0.f;
                }
            }
        };
        float4 cur[4], next[4];
        const int64_t b0 = ((lo + skip) & ~(int64_t)3) - skip;      // at a boundary, at most 3 before lo
        load(b0, next);
        for (int64_t b = b0; b < hi; b += 512) {
#pragma unroll
            for (int q = 0; q < 4; ++q) cur[q] = next[q];
            if (b + 512 < hi) load(b + 512, next);
            unsigned in = __ballot_sync(0xffffffffu, lane < R && win + K > b && win < b + 512);
            while (in) {                                            // diagonals inside the stretch
                const int l = __ffs(in) - 1;
                in &= in - 1;
                const int d = (int)(__shfl_sync(0xffffffffu, win, l) - b) - 4 * lane;    // from this lane's first value
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    if ((unsigned)(128 * q - d) < (unsigned)K) cur[q].x = 0.f;
                    if ((unsigned)(128 * q + 1 - d) < (unsigned)K) cur[q].y = 0.f;
                    if ((unsigned)(128 * q + 2 - d) < (unsigned)K) cur[q].z = 0.f;
                    if ((unsigned)(128 * q + 3 - d) < (unsigned)K) cur[q].w = 0.f;
                }
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const float v[4] = {cur[q].x, cur[q].y, cur[q].z, cur[q].w};
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    const float p = v[c] * v[c];
                    acc[q] = df_add(acc[q], DF{p, fmaf(v[c], v[c], -p)});
                }
            }
        }
    }
    DF sum = df_add(df_add(acc[0], acc[1]), df_add(acc[2], acc[3]));
    for (int d = 16; d > 0; d >>= 1) {
        const DF o{__shfl_xor_sync(0xffffffffu, sum.hi, d), __shfl_xor_sync(0xffffffffu, sum.lo, d)};
        sum = df_add(sum, o);
    }
    if (lane == 0) red[wid] = (double)sum.hi + (double)sum.lo;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int k = 0; k < kSumsqThreads / 32; ++k) t += red[k];
        partial[blockIdx.x] = t;
    }
    if (blockIdx.x == 0 && threadIdx.x >= gridDim.x && threadIdx.x < kSumsqBlocks) partial[threadIdx.x] = 0.0;
}

// sc = (2^s, 2^-s, 2^r, 2^-r) from the sum of squares F^2 (the kSumsqBlocks
// partials, added as a tree) and, when given, the largest squared norm of the K
// vectors (else the vectors have norm 1), with F ||x|| < 2^e and ||x|| < 2^ex:
//   s = min(60 - e, 124 - ex): the mirrored products' units 2^-s keep every
//       accumulator below 2^60, and every x_i 2^s is an FP32 pair;
//   r = 1 - ex: the row part multiplies x 2^r, of norm below 2 (0 when the
//       vectors have norm 1).
__global__ void __launch_bounds__(kSumsqBlocks) k_mirror_scale(const double *partial, int K, const double *xn2, double *sc)
{
    __shared__ double red[kSumsqBlocks];
    const int tid = threadIdx.x;
    red[tid] = partial[tid];
    __syncthreads();
    for (int d = kSumsqBlocks / 2; d > 0; d >>= 1) {              // the order upper_sumsq adds in
        if (tid < d) red[tid] += red[tid + d];
        __syncthreads();
    }
    if (tid != 0) return;
    const double f2 = red[0];
    double m = 1.0;
    if (xn2) {
        m = 0.0;
        for (int k = 0; k < K; ++k) m = fmax(m, xn2[k]);
    }
    int e = 0, ex = 1;
    if (f2 > 0.0 && m > 0.0) (void)frexp(sqrt(f2 * m) * (1.0 + 1e-6), &e);
    if (xn2 && m > 0.0) (void)frexp(sqrt(m) * (1.0 + 1e-6), &ex);
    const int sh = min(60 - e, 124 - ex), r = xn2 ? 1 - ex : 0;
    sc[0] = ldexp(1.0, sh);
    sc[1] = ldexp(1.0, -sh);
    sc[2] = ldexp(1.0, r);
    sc[3] = ldexp(1.0, -r);
}

// The GPU's FP64 units are few, so the product runs in FP32 pairs: x is
// split once per product into hi + lo floats (xs), a product v (hi + lo) is
// the pair (v hi, fma(v, hi, -v hi) + v lo) (about 47 bits), row sums are
// double-float sums, and a mirrored product goes to the fixed-point
// accumulator as the rounded hi plus the rounded lo (at most 1 unit of
// error).  No FP64 operation runs per stored nonzero.
__device__ __forceinline__ float2 split2(double v)
{
    const float h = (float)v;
    return make_float2(h, (float)(v - (double)h));
}

__device__ __forceinline__ DF df_prod(float v, float2 x)
{
    const float p = v * x.x;
    return DF{p, fmaf(v, x.y, fmaf(v, x.x, -p))};
}

// f rounded to the nearest integer (halves away from zero) by integer
// operations on its bits; |f| < 2^62.  (The hardware's 64-bit conversions run
// on the FP64 units.)
__device__ __forceinline__ long long round_ll(float f)
{
    const unsigned b = __float_as_uint(f);
    const int sh = (int)((b >> 23) & 0xFFu) - 150;                 // |f| = m 2^sh
    const unsigned m = (b & 0x7FFFFFu) | 0x800000u;
    long long v = 0;                                                // |f| < 0.5, zero, subnormal
    if (sh >= 0) v = (long long)m << sh;
    else if (sh >= -24) v = (long long)((m + (1u << (-sh - 1))) >> -sh);
    return (b >> 31) ? -v : v;
}

// x rounded to the nearest integer, halves away from zero as round_ll (the half is
// added rounding towards zero: a sum just below an integer must not reach it)
__device__ __forceinline__ int round_i32(float x)
{
    return __float2int_rz(__fadd_rz(x, copysignf(0.5f, x)));
}

// The mirrored product q (hi + lo, units 2^-s) as an integer: hi and lo each
// rounded.  Below 2^50 hi splits exactly into A 2^30 + rem, |rem| <= 2^29 (A through
// the float's own rounding at 1.5 2^23, rem by one FMA; from 2^24 on hi is an
// integer, so rounding rem rounds hi), and |lo| <= 1.5 2^26 (v x.y, and half the last
// bit of hi): the sum of both fits 32 bits.  Two 32-bit conversions
// and a wide multiply-add, some 16 instructions, where shifting the two mantissas
// took about 40: a call of 64 sets at 3+4 Nmax=4 2.69 -> 2.44 ms, at 4+4 Nmax=4
// 8.05 -> 7.33 ms; one set, bound by its atomic adds, unchanged.
__device__ __forceinline__ void mirror_add(unsigned long long *a, DF q)
{
    long long v;
    if (fabsf(q.hi) < 1125899906842624.f) {
        const float t = fmaf(q.hi, 9.31322574615478515625e-10f, 12582912.f);         // hi 2^-30
        const float rem = fmaf(t - 12582912.f, -1073741824.f, q.hi);
        v = (long long)(__float_as_int(t) - 0x4B400000) * 1073741824ll + (round_i32(rem) + round_i32(q.lo));
    } else {
        v = round_ll(q.hi) + round_ll(q.lo);
    }
    atomicAdd(a, (unsigned long long)v);
}

// xs[t] = x[t] 2^r (the row part's factor) and xm[t] = x[t] 2^s (the
// mirrored products'), each as hi + lo floats
__global__ void k_split(int64_t n, const double *x, const double *sc, float2 *xs, float2 *xm)
{
    const double fr = sc[2], fs = sc[0];
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n; t += (int64_t)gridDim.x * blockDim.x) {
        const double v = x[t];
        xs[t] = split2(v * fr);
        xm[t] = split2(v * fs);
    }
}

// K > 16: lanes over sets, two per lane per pass; K <= 16 (KS = next power
// of two): 32/KS lane groups split the row's nonzeros, four at a time per
// group, and the groups' row sums are reduced at the end, and the
// matrix is read with evict-first loads, so that its stream does not push x
// and the accumulators out of L2 (with lanes over sets the same hint ran
// slower).  Each block walks
// one contiguous run of `per` rows, so that rows of one proton sub-determinant
// (which touch the same x and accumulator blocks) share its L1.
template <int KS>
__global__ void __launch_bounds__(kThreads, 4) k_spmv(RowRange rr, int K, const int64_t *rowptr, const int32_t *col, const float *vem,
                       const float2 *xs, const float2 *xm, float2 *yrow, unsigned long long *yfix, int64_t per)
{
    const int lane = threadIdx.x & 31;
    const int64_t r0 = rr.r0 + blockIdx.x * per, r1 = min(rr.r1, r0 + per);
    const int wpb = blockDim.x >> 5;
    for (int64_t i = r0 + (threadIdx.x >> 5); i < r1; i += wpb) {
        const int64_t a0 = rowptr[i] - rr.base, a1 = rowptr[i + 1] - rr.base;
        if (KS >= 32) {
            const int KK = KS == 64 ? 64 : K;                      // KS = 64: exactly 64 sets
            for (int s0 = 0; s0 < KK; s0 += 64) {
                const int sa = s0 + lane, sb = s0 + 32 + lane;
                const bool ha = sa < KK, hb = sb < KK;
                const float2 Xa = ha ? xm[i * KK + sa] : make_float2(0.f, 0.f);
                const float2 Xb = hb ? xm[i * KK + sb] : make_float2(0.f, 0.f);
                DF acc_a = df_of(0.f), acc_b = df_of(0.f);
                int64_t k = a0;
                for (; k + 3 < a1; k += 4) {
                    int64_t c[4];
                    float va[4], vb[4];
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        c[u] = col[k + u];
                        va[u] = ha ? vem[(k + u) * KK + sa] : 0.f;
                        vb[u] = hb ? vem[(k + u) * KK + sb] : 0.f;
                    }
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        if (ha) acc_a = df_add(acc_a, df_prod(va[u], xs[c[u] * KK + sa]));
                        if (hb) acc_b = df_add(acc_b, df_prod(vb[u], xs[c[u] * KK + sb]));
                        if (c[u] != i) {
                            if (ha) mirror_add(yfix + c[u] * KK + sa, df_prod(va[u], Xa));
                            if (hb) mirror_add(yfix + c[u] * KK + sb, df_prod(vb[u], Xb));
                        }
                    }
                }
                for (; k < a1; ++k) {
                    const int64_t c = col[k];
                    const float va = ha ? vem[k * KK + sa] : 0.f, vb = hb ? vem[k * KK + sb] : 0.f;
                    if (ha) acc_a = df_add(acc_a, df_prod(va, xs[c * KK + sa]));
                    if (hb) acc_b = df_add(acc_b, df_prod(vb, xs[c * KK + sb]));
                    if (c != i) {
                        if (ha) mirror_add(yfix + c * KK + sa, df_prod(va, Xa));
                        if (hb) mirror_add(yfix + c * KK + sb, df_prod(vb, Xb));
                    }
                }
                if (ha) yrow[i * KK + sa] = make_float2(acc_a.hi, acc_a.lo);
                if (hb) yrow[i * KK + sb] = make_float2(acc_b.hi, acc_b.lo);
            }
        } else {
            constexpr int G = 32 / KS;
            const int g = lane / KS, s = lane % KS;
            DF acc = df_of(0.f);
            if (s < K) {
                const float2 Xi = xm[i * K + s];
                int64_t k = a0 + g;
                for (; k + 3 * G < a1; k += 4 * G) {
                    int64_t c[4];
                    float v[4];
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        c[u] = __ldcs(col + k + u * G);
                        v[u] = __ldcs(vem + (k + u * G) * K + s);
                    }
                    float2 xj[4];
#pragma unroll
                    for (int u = 0; u < 4; ++u) xj[u] = xs[c[u] * K + s];
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        acc = df_add(acc, df_prod(v[u], xj[u]));
                        if (c[u] != i) mirror_add(yfix + c[u] * K + s, df_prod(v[u], Xi));
                    }
                }
                for (; k < a1; k += G) {
                    const int64_t c = __ldcs(col + k);
                    const float v = __ldcs(vem + k * K + s);
                    acc = df_add(acc, df_prod(v, xs[c * K + s]));
                    if (c != i) mirror_add(yfix + c * K + s, df_prod(v, Xi));
                }
            }
            for (int d = 16; d >= KS; d >>= 1) {
                const DF o{__shfl_xor_sync(0xffffffffu, acc.hi, d), __shfl_xor_sync(0xffffffffu, acc.lo, d)};
                acc = df_add(acc, o);
            }
            if (g == 0 && s < K) yrow[i * K + s] = make_float2(acc.hi, acc.lo);
        }
    }
}

// y = row part 2^-r + mirrored part 2^-s; the accumulator is cleared for the
// next product
__device__ __forceinline__ double finish_entry(const float2 *yrow, unsigned long long *yfix, int64_t t, double sinv, double rinv)
{
    const float2 r = yrow[t];
    const double y = ((double)r.x + (double)r.y) * rinv + (double)(long long)yfix[t] * sinv;
    yfix[t] = 0ull;
    return y;
}

__global__ void k_sym_finish(int64_t n, const double *sc, const float2 *yrow, double *y, unsigned long long *yfix)
{
    const double sinv = sc[1], rinv = sc[3];
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n; t += (int64_t)gridDim.x * blockDim.x)
        y[t] = finish_entry(yrow, yfix, t, sinv, rinv);
}

// Row shards: the local rows' row part in FP64 into yx (the other entries
// stay 0, so that a sum over the shards is exact); then, once the caller has
// summed yx and the accumulators over the shards, y = yx + acc 2^-s and both
// are cleared.  The same operations in the same order as k_sym_finish.
__global__ void k_shard_rows(RowRange rr, int K, const double *sc, const float2 *yrow, double *yx)
{
    const double rinv = sc[3];
    const int64_t n = (rr.r1 - rr.r0) * K, o = rr.r0 * K;
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n; t += (int64_t)gridDim.x * blockDim.x) {
        const float2 r = yrow[o + t];
        yx[o + t] = ((double)r.x + (double)r.y) * rinv;
    }
}

__global__ void k_shard_finish(int64_t n, const double *sc, double *yx, unsigned long long *acc, double *y)
{
    const double sinv = sc[1];
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n; t += (int64_t)gridDim.x * blockDim.x) {
        y[t] = yx[t] + (double)(long long)acc[t] * sinv;
        yx[t] = 0.0;
        acc[t] = 0ull;
    }
}

// Rows a block of the product takes, a multiple of its 8 warps.  Long runs share more
// of L1, short ones leave the GPU less idle at the end, and the more sets, the
// longer a row takes.  Measured, us a call, by rows a block (and, last, for 4,864
// blocks of equal runs, whose 8 warps share 11, 30, 42 or 456 rows unevenly):
//   one set:  4+4 Nmax=6   32: 5925  64: 5673  128: 5589  192: 5634   5998
//             5+6 Nmax=4   32: 1457  64: 1414  128: 1432  192: 1472   1451
//             4+4 Nmax=4   16:  325  32:  316   64:  322               314
//   4 sets:   3+3 Nmax=6    8: 1072  16: 1053   32: 1110              1155
//   8 sets:   5+6 Nmax=4    8: 6259  16: 6178   32: 6117   64: 6280   6912
//   32 sets:  4+4 Nmax=4    8: 4986  16: 5139   32: 5512              5465
//   64 sets:  3+4 Nmax=4    8: 1811  16: 1893   32: 2248              1975
inline int64_t rows_per_block(int64_t rows, int K)
{
    const int64_t per = (rows + 4 * 4864 * (int64_t)K) / (8 * 4864 * (int64_t)K) * 8;
    return std::max<int64_t>(8, std::min<int64_t>(per, std::max(16, 128 / K)));
}

// One product's k_spmv launch.  (Passes of 32 sets, to keep a share of the
// randomly accessed vectors L2-resident at 64 sets, ran slower.)
void launch_spmv(RowRange rr, int K, const int64_t *rowptr, const int32_t *col, const float *vem, const float2 *xs,
                 const float2 *xm, float2 *yrow, unsigned long long *yfix, cudaStream_t st)
{
    const int64_t rows = rr.r1 - rr.r0, per = rows_per_block(rows, K);
    const int64_t blocks = (rows + per - 1) / per;              // rows < 2^31: at most 2^28
    if (blocks == 0) return;
    const unsigned gr = (unsigned)blocks;
    count_launches(1);
    if (K == 64) k_spmv<64><<<gr, kThreads, 0, st>>>(rr, K, rowptr, col, vem, xs, xm, yrow, yfix, per);
    else if (K > 16) k_spmv<32><<<gr, kThreads, 0, st>>>(rr, K, rowptr, col, vem, xs, xm, yrow, yfix, per);
    else if (K == 1) k_spmv<1><<<gr, kThreads, 0, st>>>(rr, K, rowptr, col, vem, xs, xm, yrow, yfix, per);
    else if (K <= 2) k_spmv<2><<<gr, kThreads, 0, st>>>(rr, K, rowptr, col, vem, xs, xm, yrow, yfix, per);
    else if (K <= 4) k_spmv<4><<<gr, kThreads, 0, st>>>(rr, K, rowptr, col, vem, xs, xm, yrow, yfix, per);
    else if (K <= 8) k_spmv<8><<<gr, kThreads, 0, st>>>(rr, K, rowptr, col, vem, xs, xm, yrow, yfix, per);
    else k_spmv<16><<<gr, kThreads, 0, st>>>(rr, K, rowptr, col, vem, xs, xm, yrow, yfix, per);
}

// ---- orthogonalisation: classical Gram-Schmidt twice, every sum in a fixed order
//
// A dot product is split over kDotBlocks blocks of kThreads threads: thread (sub,
// s) of block b takes rows b per + sub, then every kDotBlocks per further on (per =
// kThreads / K rows a block, sets s); the block's threads are added in
// order, then the blocks in order.  That order is part of the results: the
// signs of the Ritz vectors hang on the last bits of the tridiagonal, so it stays
// whatever executes it.  What is fast here: a block takes 32 vectors, whose
// ordered adds run side by side in one warp (an FP64 instruction occupies the
// SM's two units for 16 cycles however few lanes are active, so one lane at a
// time made the adds, not the memory, the limit); they run from shared memory,
// the blocks' sums are loaded together before theirs, and blocks and threads
// without rows (whose sums are zeros) are left out.  (A thread adding 256 values
// of one vector per block, and again 256 blocks' sums from global memory, took 73
// + 17 us for the dot products of a step at 800 rows, three times a step.)
constexpr int kDotVecs = 32;           // most vectors of a block (dot_vecs)
constexpr int kDotPad = kThreads + 1;  // (the ordered adds read a column of 32 vectors: no bank twice)

__host__ __device__ inline int dot_blocks(int64_t dim, int K)
{
    const int64_t per = kThreads / K, n = (dim + per - 1) / per;
    return (int)(n < 1 ? 1 : n < kDotBlocks ? n : kDotBlocks);
}

// partial[blk * nvec * K + r * K + s] = block blk's part of sum_i V[r][i][s] w[i][s]
template <int KC>
__global__ void __launch_bounds__(kThreads) k_dots(int64_t dim, int K_, int nvec, const double *V, int64_t vstride,
                                                   const double *w, double *partial, int vecs)
{
    extern __shared__ double red[];                               // min(vecs, nvec) x kDotPad
    const int K = KC ? KC : K_, per = kThreads / K, tid = threadIdx.x;
    const int s = KC == 1 ? 0 : tid % K, sub = KC == 1 ? tid : tid / K;
    const int r0 = blockIdx.y * vecs, nv = min(vecs, nvec - r0);
    const int64_t i0 = (int64_t)blockIdx.x * per + sub, step = (int64_t)kDotBlocks * per;
    for (int u0 = 0; u0 < nv; u0 += 4) {
        double acc[4] = {0.0, 0.0, 0.0, 0.0};
        const double *v = V + (int64_t)(r0 + u0) * vstride + s;
        if (sub < per && u0 + 4 <= nv) {
#pragma unroll 4
            for (int64_t i = i0; i < dim; i += step) {
                const double x = w[i * K + s];
#pragma unroll
                for (int u = 0; u < 4; ++u) acc[u] += v[u * vstride + i * K] * x;
            }
        } else if (sub < per) {
#pragma unroll 2
            for (int64_t i = i0; i < dim; i += step) {
                const double x = w[i * K + s];
#pragma unroll
                for (int u = 0; u < 3; ++u)
                    if (u0 + u < nv) acc[u] += v[u * vstride + i * K] * x;
            }
        }
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (u0 + u < nv) red[(u0 + u) * kDotPad + tid] = acc[u];
    }
    __syncthreads();
    const int rows = (int)min((int64_t)per, dim - (int64_t)blockIdx.x * per);       // threads with rows
    for (int q = tid; q < nv * K; q += kThreads) {
        const int u = KC == 1 ? q : q / K, ss = KC == 1 ? 0 : q - u * K;
        const double *o = red + u * kDotPad + ss;
        double t = 0.0;
#pragma unroll 8
        for (int x = 0; x < rows; ++x) t += o[x * K];
        partial[(int64_t)blockIdx.x * nvec * K + (r0 + u) * K + ss] = t;
    }
}

// What k_dots_sum does with the sums t over the blocks, q = r K + s:
//   h    store them (coefficients of the next update); alpha[s] gets the last
//        vector's, added to its value of the first pass in the second
//   beta |w|^2 to beta[s], f[s] = 1 / |w|, or 0 for a set that is done or whose
//        Krylov space is exhausted (the host's test for that)
//   unit store them, f[s] = 1 / sqrt(t) (0 for a zero vector)
enum { kSumFirst = 0, kSumSecond = 1, kSumBeta = 2, kSumUnit = 3 };
constexpr int kSumRows = 128;

__global__ void __launch_bounds__(kThreads) k_dots_sum(int mode, int nvec, int K, int blocks, const double *partial, double *out,
                                                       double *alpha, double *beta, double *f, const int *done)
{
    __shared__ double red[kSumRows][33];
    const int nq = nvec * K, lane = threadIdx.x & 31, q = blockIdx.x * 32 + lane;
    double t = 0.0;
    for (int b0 = 0; b0 < blocks; b0 += kSumRows) {
        const int n = min(kSumRows, blocks - b0);
        if (q < nq)
            for (int b = threadIdx.x >> 5; b < n; b += kThreads / 32) red[b][lane] = partial[(int64_t)(b0 + b) * nq + q];
        __syncthreads();
        if (threadIdx.x < 32 && q < nq) {
#pragma unroll 8
            for (int b = 0; b < n; ++b) t += red[b][lane];
        }
        __syncthreads();
    }
    if (threadIdx.x >= 32 || q >= nq) return;
    const int s = q % K, r = q / K;
    if (mode == kSumFirst || mode == kSumSecond) {
        out[q] = t;
        if (r == nvec - 1) alpha[s] = mode == kSumFirst ? t : alpha[s] + t;
    } else if (mode == kSumBeta) {
        beta[s] = t;
        const double b = sqrt(fmax(t, 0.0));
        f[s] = done[s] || b <= 1e-12 * (fabs(alpha[s]) + 1.0) ? 0.0 : 1.0 / b;
    } else {
        out[q] = t;
        f[s] = t > 0.0 ? 1.0 / sqrt(t) : 0.0;
    }
}

// w[i][s] -= sum_r h[r][s] V[r][i][s], r ascending (out: sum_r h[r][s] V[r][i][s]
// from zero); eight loads in flight
template <bool SUB>
__global__ void __launch_bounds__(kThreads) k_combine(int64_t n, int K, int nvec, const double *V, int64_t vstride, const double *h,
                                                      double *w)
{
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n; t += (int64_t)gridDim.x * blockDim.x) {
        const double *v = V + t, *c = h + (K == 1 ? 0 : t % K);
        double x = SUB ? w[t] : 0.0;
        int r = 0;
        for (; r + 8 <= nvec; r += 8) {
            double y[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) y[u] = v[(int64_t)(r + u) * vstride];
#pragma unroll
            for (int u = 0; u < 8; ++u) x = SUB ? x - c[(r + u) * K] * y[u] : x + c[(r + u) * K] * y[u];
        }
        for (; r < nvec; ++r) x = SUB ? x - c[r * K] * v[(int64_t)r * vstride] : x + c[r * K] * v[(int64_t)r * vstride];
        w[t] = x;
    }
}

// v = w f, the next Lanczos vector, and its split for the product (k_split)
__global__ void k_next(int64_t n, int K, const double *w, const double *f, const double *sc, double *v, float2 *xs, float2 *xm)
{
    const double fr = sc[2], fs = sc[0];
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n; t += (int64_t)gridDim.x * blockDim.x) {
        const double x = w[t] * f[K == 1 ? 0 : t % K];
        v[t] = x;
        xs[t] = split2(x * fr);
        xm[t] = split2(x * fs);
    }
}

// deterministic start vector: 1 + 0.5 u_i, u_i from the splitmix64 hash of i (same for every set)
__global__ void k_start(int64_t dim, int K, double *v)
{
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < dim * K; t += (int64_t)gridDim.x * blockDim.x) {
        unsigned long long z = (unsigned long long)(t / K) + 0x9E3779B97F4A7C15ull;
        z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
        z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
        z ^= z >> 31;
        v[t] = 1.0 + 0.5 * (double)(z >> 11) * (1.0 / 9007199254740992.0);
    }
}

// evec[s * dim + i] = w[i * K + s] f[s]  (set-major output)
__global__ void k_ritz_out(int64_t dim, int K, const double *w, const double *f, double *evec)
{
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < dim * K; t += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i = t / K;
        const int s = (int)(t - i * K);
        evec[(int64_t)s * dim + i] = w[t] * f[s];
    }
}

// Vectors of a block of k_dots: as many as leave two blocks per SM, in fours;
// four where a block has few ordered adds (many sets) or short vectors leave few
// blocks.  One size for all, at 800 rows / 143,792 rows / 48,917 rows of 64 sets,
// a whole solve: 4 vectors 3.87 / 47.5 / 383 ms, 32 vectors 4.41 / 38.3 / 391 ms.
int dot_vecs(int nb, int K, int nvec)
{
    if (K >= 16) return 4;
    return std::max(4, std::min(kDotVecs, nb * nvec / 304 / 4 * 4));
}

// k_dots takes up to 66 KB of shared memory (set once per device; idempotent).  The set
// count is fixed at compile time for 64 sets, the batched configuration, as in k_spmv (a
// solve of 64 sets of 3+4 Nmax=4 takes 328 ms without, 325 with), and for one.
cudaError_t prepare_dots(int K)
{
    const int bytes = (int)sizeof(double) * kDotPad * kDotVecs;
    const void *f = K == 1 ? (const void *)k_dots<1> : K == 64 ? (const void *)k_dots<64> : (const void *)k_dots<0>;
    return cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
}

// sums[q] over r < nvec of V[r] . w per set, then `mode` (k_dots_sum)
void launch_dots(int mode, int64_t dim, int K, int nvec, const double *V, int64_t vstride, const double *w, double *partial,
                 double *out, double *alpha, double *beta, double *f, const int *done, cudaStream_t st)
{
    const int nb = dot_blocks(dim, K);
    const int vecs = dot_vecs(nb, K, nvec);
    const dim3 grid(nb, (nvec + vecs - 1) / vecs);
    const size_t smem = sizeof(double) * kDotPad * std::min(nvec, vecs);
    count_launches(2);
    if (K == 1) k_dots<1><<<grid, kThreads, smem, st>>>(dim, K, nvec, V, vstride, w, partial, vecs);
    else if (K == 64) k_dots<64><<<grid, kThreads, smem, st>>>(dim, K, nvec, V, vstride, w, partial, vecs);
    else k_dots<0><<<grid, kThreads, smem, st>>>(dim, K, nvec, V, vstride, w, partial, vecs);
    k_dots_sum<<<(nvec * K + 31) / 32, kThreads, 0, st>>>(mode, nvec, K, nb, partial, out, alpha, beta, f, done);
}

int grid_for(int64_t n)
{
    return (int)std::max<int64_t>(1, std::min<int64_t>((n + kThreads - 1) / kThreads, 152 * 16));
}

}  // namespace

int64_t lanczos_bytes(int64_t dim, int64_t nnz, int K, int max_iter)
{
    const int64_t m = std::min<int64_t>(max_iter, dim);
    int64_t bytes = 8 * (m + 1) * dim * K + 8 * dim * K;            // Lanczos vectors, w
    bytes += 32 * dim * K;                                          // mirror accumulators, split x, row part
    bytes += 8 * (m + 1) * K * kDotBlocks;   // partial sums
    bytes += 8 * (m + 1) * K + 64 * K + 32;                         // coefficients, scalars, scale
    if (K > 1) bytes += 4 * nnz * K;                                // element-major values
    return bytes + 8 * 256;                                         // allocation granules
}

// Page-locked blocks for the two scalars a set returns per step (two steps in
// flight) and the done flags, kept for the next call; at most kKeep of them.
struct StepLog {
    static constexpr int kMaxSets = 256, kKeep = 16;
    double *p = nullptr;                                            // [2][2 K], then int done[K]
    static std::mutex &mu() { static std::mutex m; return m; }
    static std::vector<double *> &kept() { static std::vector<double *> v; return v; }
    bool get()
    {
        {
            std::lock_guard<std::mutex> lock(mu());
            if (!kept().empty()) {
                p = kept().back();
                kept().pop_back();
                return true;
            }
        }
        if (cudaHostAlloc((void **)&p, sizeof(double) * 4 * kMaxSets + sizeof(int) * kMaxSets, cudaHostAllocPortable) != cudaSuccess) {
            (void)cudaGetLastError();
            p = nullptr;
        }
        return p != nullptr;
    }
    ~StepLog()                                                      // the caller has synchronised the copies
    {
        if (!p) return;
        std::lock_guard<std::mutex> lock(mu());
        if ((int)kept().size() < kKeep) kept().push_back(p);
        else cudaFreeHost(p);
    }
    double *slot(int j, int K) const { return p + (j & 1) * 2 * K; }
    int *done() const { return reinterpret_cast<int *>(p + 4 * kMaxSets); }
};

// sh->f2 -> (2^s, 2^-s, 1, 1): the scale k_mirror_scale gives unit vectors
static void shard_scale(double f2, double *sc)
{
    int e = 0;
    if (f2 > 0.0) (void)std::frexp(std::sqrt(f2) * (1.0 + 1e-6), &e);
    const int sh = std::min(60 - e, 124 - 1);
    sc[0] = std::ldexp(1.0, sh);
    sc[1] = std::ldexp(1.0, -sh);
    sc[2] = sc[3] = 1.0;
}

int lanczos(const cih_basis &b, const int64_t *rowptr, const int32_t *col, const float *val, int K, int nev,
            int max_iter, double tol, double *evals, double *evec0, cudaStream_t st, bool values_em,
            const ShardRun *sh)
{
    const int64_t dim = b.dim;
    for (int k = 0; k < K * nev; ++k) evals[k] = NAN;
    if (dim == 0) return CIH_OK;
    if (K > kThreads) return fail(CIH_ERR_UNSUPPORTED, "lanczos: at most 256 sets per call");
    if (dim > INT32_MAX) return fail(CIH_ERR_UNSUPPORTED, "lanczos: dimension above 2^31");
    // the rows this process multiplies, and the stored nonzeros its arrays hold
    const int64_t r0 = sh ? sh->r0 : 0, r1 = sh ? sh->r1 : dim;
    int64_t ends[2] = {0, 0};
    cudaError_t e = cudaMemcpyAsync(&ends[0], rowptr + r0, sizeof(int64_t), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaMemcpyAsync(&ends[1], rowptr + r1, sizeof(int64_t), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return cuda_fail(e, "lanczos: read nnz");
    const int64_t base = sh ? ends[0] : 0, nnz = ends[1] - base;
    const RowRange rr{r0, r1, base};
    const int m_max = (int)std::min<int64_t>(max_iter, dim);
    const int64_t vstride = dim * K;

    std::vector<void *> bufs;
    auto alloc = [&](void **p, size_t bytes) -> bool {
        if (cudaMallocFromPoolAsync(p, std::max<size_t>(bytes, 16), b.pool, st) != cudaSuccess) {
            (void)cudaGetLastError();
            return false;
        }
        bufs.push_back(*p);
        return true;
    };
    float *vem = nullptr;
    unsigned long long *yfix = nullptr;
    float2 *xs = nullptr, *xm = nullptr, *yrow = nullptr;
    double *V = nullptr, *w = nullptr, *partial = nullptr, *hdev = nullptr, *slog = nullptr, *fdev = nullptr, *sc = nullptr;
    int *ddone = nullptr;
    bool ok = (sh ? (yfix = sh->acc) != nullptr : alloc((void **)&yfix, sizeof(unsigned long long) * (size_t)vstride)) &&
              alloc((void **)&xs, sizeof(float2) * (size_t)vstride) &&
              alloc((void **)&xm, sizeof(float2) * (size_t)vstride) &&
              alloc((void **)&yrow, sizeof(float2) * (size_t)vstride) &&
              alloc((void **)&V, sizeof(double) * (size_t)(m_max + 1) * vstride) &&
              alloc((void **)&w, sizeof(double) * vstride) &&
              alloc((void **)&partial, sizeof(double) * (size_t)(m_max + 1) * K * kDotBlocks) &&
              alloc((void **)&hdev, sizeof(double) * (size_t)(m_max + 1) * K) &&
              alloc((void **)&slog, sizeof(double) * 4 * K) && alloc((void **)&fdev, sizeof(double) * K) &&
              alloc((void **)&sc, sizeof(double) * 4) && alloc((void **)&ddone, sizeof(int) * K);
    if (ok && K > 1 && !values_em) ok = alloc((void **)&vem, sizeof(float) * (size_t)nnz * K);
    StepLog pin;
    cudaEvent_t ev[2] = {nullptr, nullptr};
    int rc = ok && pin.get() ? CIH_OK : fail(CIH_ERR_NOMEM, "lanczos: memory");
    for (int i = 0; i < 2 && !rc; ++i)
        if ((e = cudaEventCreateWithFlags(&ev[i], cudaEventDisableTiming)) != cudaSuccess) rc = cuda_fail(e, "lanczos: event");
    if (!rc && (e = prepare_dots(K)) != cudaSuccess) rc = cuda_fail(e, "lanczos: shared memory");
    const int g = grid_for(vstride);

    // element-major values, the mirror scale and cleared accumulators (no host
    // synchronisation; a shard's scale comes from the whole matrix's norm)
    if (!rc) {
        if (K > 1 && !values_em) {
            count_launches(1);
            k_vals_em<<<grid_for(nnz * K), kThreads, 0, st>>>(K, nnz, val, vem);
        } else {
            vem = const_cast<float *>(val);                         // K = 1, or already element-major
        }
        cudaMemsetAsync(ddone, 0, sizeof(int) * K, st);
        if (sh) {
            double hsc[4];
            shard_scale(sh->f2, hsc);
            e = cudaMemcpyAsync(sc, hsc, sizeof(hsc), cudaMemcpyHostToDevice, st);
            if (e == cudaSuccess) e = cudaStreamSynchronize(st);
            if (e != cudaSuccess) rc = cuda_fail(e, "lanczos: shard scale");
        } else {
            cudaMemsetAsync(yfix, 0, sizeof(unsigned long long) * (size_t)vstride, st);
            count_launches(2);
            k_upper_sumsq<<<kSumsqGrid, kSumsqThreads, 0, st>>>(rr, K, rowptr, vem, partial);
            k_mirror_scale<<<1, kSumsqBlocks, 0, st>>>(partial, K, nullptr, sc);
        }
    }

    // w = H v_j from the split of v_j
    auto spmv = [&]() -> int {
        launch_spmv(rr, K, rowptr, col, vem, xs, xm, yrow, yfix, st);
        if (!sh) {
            count_launches(1);
            k_sym_finish<<<g, kThreads, 0, st>>>(vstride, sc, yrow, w, yfix);
            return CIH_OK;
        }
        // a shard: its rows' row part, then the caller sums both buffers over the shards
        count_launches(2);
        k_shard_rows<<<grid_for((r1 - r0) * K), kThreads, 0, st>>>(rr, K, sc, yrow, sh->yx);
        cudaError_t ee = cudaStreamSynchronize(st);
        if (ee != cudaSuccess) return cuda_fail(ee, "lanczos: shard product");
        if (sh->combine(sh->ctx) != 0) return fail(CIH_ERR_ARG, "lanczos: the shard combine callback failed");
        k_shard_finish<<<g, kThreads, 0, st>>>(vstride, sc, sh->yx, yfix, w);
        return CIH_OK;
    };

    // v0 = start / |start| per set
    if (!rc) {
        count_launches(2);
        k_start<<<g, kThreads, 0, st>>>(dim, K, w);
        launch_dots(kSumUnit, dim, K, 1, w, vstride, w, partial, hdev, nullptr, nullptr, fdev, nullptr, st);
        k_next<<<g, kThreads, 0, st>>>(vstride, K, w, fdev, sc, V, xs, xm);
    }
    // step j on the device: product, orthogonalisation, the scalars to the host,
    // and the next vector (a finished set's is zero)
    auto enqueue = [&](int j) -> int {
        const int r = spmv();
        if (r) return r;
        double *alpha = slog + (j & 1) * 2 * K, *beta = alpha + K;
        for (int pass = 0; pass < 2; ++pass) {                      // alpha_j = v_j . H v_j (+ the second pass's small correction)
            launch_dots(pass ? kSumSecond : kSumFirst, dim, K, j + 1, V, vstride, w, partial, hdev, alpha, nullptr, nullptr, nullptr, st);
            count_launches(1);
            k_combine<true><<<g, kThreads, 0, st>>>(vstride, K, j + 1, V, vstride, hdev, w);
        }
        launch_dots(kSumBeta, dim, K, 1, w, vstride, w, partial, nullptr, alpha, beta, fdev, ddone, st);
        cudaMemcpyAsync(pin.slot(j, K), alpha, sizeof(double) * 2 * K, cudaMemcpyDeviceToHost, st);
        cudaEventRecord(ev[j & 1], st);
        if (j + 1 < m_max) {
            count_launches(1);
            k_next<<<g, kThreads, 0, st>>>(vstride, K, w, fdev, sc, V + (int64_t)(j + 1) * vstride, xs, xm);
        }
        const cudaError_t ee = cudaGetLastError();
        return ee == cudaSuccess ? CIH_OK : cuda_fail(ee, "lanczos kernels");
    };
    // The device runs one step ahead: step j + 1 is queued before the host reads
    // step j's scalars and decides whether the sets have converged, so the
    // tridiagonal solves cost no device time; the last step queued may be unused.
    // (Over shards the caller's callback runs in every step: no step ahead.)
    std::vector<std::vector<double>> alpha(K), beta(K);
    std::vector<int> done(K, 0), m_of(K, 0), met(K, 0);
    std::vector<double> theta((size_t)K * nev, NAN), warm(K, NAN);
    int m = 0;
    if (!rc && m_max > 0) rc = enqueue(0);
    for (int j = 0; j < m_max && !rc; ++j) {
        if (!sh && j + 1 < m_max && (rc = enqueue(j + 1))) break;
        if ((e = cudaEventSynchronize(ev[j & 1])) != cudaSuccess) { rc = cuda_fail(e, "lanczos: step"); break; }
        const double *log = pin.slot(j, K);
        m = j + 1;
        // per set (sets in parallel on host threads): Ritz values and residual
        // bounds beta_m |z_m| of the lowest nev, from the tridiagonal's QR
        // eigen-decomposition (last eigenvector components); while the nev-th
        // pair alone is far from its bound, the decomposition is left out
        parallel_sets(K, [&](int s) {
            if (done[s]) return;
            const double bj = std::sqrt(std::max(log[K + s], 0.0));
            alpha[s].push_back(log[s]);
            beta[s].push_back(bj);
            const int ms = m_of[s] = (int)alpha[s].size();
            const int nv = std::min(nev, ms);
            bool conv = ms >= std::min<int64_t>(nev, dim);
            const bool invariant = bj <= 1e-12 * (std::fabs(alpha[s].back()) + 1.0);
            if (!invariant && ms < m_max && (!conv || tridiag_pair_open(ms, alpha[s].data(), beta[s].data(), nv - 1, bj,
                                                                        10.0 * tol, warm[s])))
                return;
            std::vector<double> dq(alpha[s]), eq(beta[s].begin(), beta[s].begin() + (ms - 1)), zl;
            if (eq.empty()) eq.push_back(0.0);
            tridiag_qr_last(ms, dq, eq, zl);
            for (int r = 0; r < nv; ++r) {
                const double th = dq[r];
                theta[(size_t)s * nev + r] = th;
                if (conv && !invariant && bj * std::fabs(zl[r]) > tol * std::max(1.0, std::fabs(th))) conv = false;
            }
            met[s] = conv || invariant;
            if (met[s] || ms == m_max) done[s] = 1;
        });
        bool all = true;
        for (int s = 0; s < K; ++s) all = all && done[s];
        if (all) break;
        if (K > 1 && !std::equal(done.begin(), done.end(), pin.done())) {
            // (the flags only spare finished sets further steps; a copy in flight may
            // carry the newer ones)
            std::copy(done.begin(), done.end(), pin.done());
            cudaMemcpyAsync(ddone, pin.done(), sizeof(int) * K, cudaMemcpyHostToDevice, st);
        }
        if (sh && j + 1 < m_max) rc = enqueue(j + 1);
    }
    int not_converged = 0;
    if (!rc) {
        std::vector<double> coef((size_t)std::max(m, 1) * K, 0.0);
        for (int s = 0; s < K; ++s) {
            const int ms = m_of[s];
            for (int r = 0; r < std::min(nev, ms); ++r) evals[(int64_t)s * nev + r] = theta[(size_t)s * nev + r];
            if (!met[s]) not_converged = 1;
            if (evec0 && ms > 0) {
                std::vector<double> z(ms);
                tridiag_eigenvector(ms, alpha[s].data(), beta[s].data(), theta[(size_t)s * nev], z.data());
                for (int r = 0; r < ms; ++r) coef[(size_t)r * K + s] = z[r];
            }
        }
        if (evec0 && m > 0) {
            // (the step queued ahead has read its coefficients before these arrive)
            cudaMemcpyAsync(hdev, coef.data(), sizeof(double) * (size_t)m * K, cudaMemcpyHostToDevice, st);
            count_launches(2);
            k_combine<false><<<g, kThreads, 0, st>>>(vstride, K, m, V, vstride, hdev, w);
            launch_dots(kSumUnit, dim, K, 1, w, vstride, w, partial, hdev, nullptr, nullptr, fdev, nullptr, st);
            k_ritz_out<<<g, kThreads, 0, st>>>(dim, K, w, fdev, evec0);
        }
    }
    e = cudaGetLastError();
    if (!rc && e != cudaSuccess) rc = cuda_fail(e, "lanczos kernels");
    for (void *p : bufs) cudaFreeAsync(p, st);
    e = cudaStreamSynchronize(st);                           // also before the page-locked block is given back
    if (!rc && e != cudaSuccess) rc = cuda_fail(e, "lanczos");
    for (cudaEvent_t x : ev)
        if (x) cudaEventDestroy(x);
    cudaMemPoolTrimTo(b.pool, kPoolKeep);                    // the Lanczos vectors go back to the system
    return rc ? rc : not_converged;
}


int ham_spmv(const cih_basis &b, const int64_t *rowptr, const int32_t *col, const float *val, int K, bool values_em,
             const double *x, double *y, cudaStream_t st)
{
    const int64_t dim = b.dim;
    if (dim == 0) return CIH_OK;
    if (K > kThreads) return fail(CIH_ERR_UNSUPPORTED, "spmv: at most 256 sets per call");
    if (dim > INT32_MAX) return fail(CIH_ERR_UNSUPPORTED, "spmv: dimension above 2^31");
    int64_t nnz = 0;
    if (K > 1 && !values_em) {
        cudaError_t e = cudaMemcpyAsync(&nnz, rowptr + dim, sizeof(int64_t), cudaMemcpyDeviceToHost, st);
        if (e == cudaSuccess) e = cudaStreamSynchronize(st);
        if (e != cudaSuccess) return cuda_fail(e, "spmv: read nnz");
    }
    const int64_t n = dim * K;
    std::vector<void *> bufs;
    auto alloc = [&](void **p, size_t bytes) -> bool {
        if (cudaMallocFromPoolAsync(p, std::max<size_t>(bytes, 16), b.pool, st) != cudaSuccess) {
            (void)cudaGetLastError();
            return false;
        }
        bufs.push_back(*p);
        return true;
    };
    unsigned long long *yfix = nullptr;
    float2 *xs = nullptr, *xm = nullptr, *yrow = nullptr;
    double *partial = nullptr, *xpart = nullptr, *xn2 = nullptr, *xf = nullptr, *sc = nullptr;
    float *vem = nullptr;
    bool ok = alloc((void **)&yfix, sizeof(unsigned long long) * (size_t)n) &&
              alloc((void **)&xs, sizeof(float2) * (size_t)n) && alloc((void **)&xm, sizeof(float2) * (size_t)n) &&
              alloc((void **)&yrow, sizeof(float2) * (size_t)n) &&
              alloc((void **)&partial, sizeof(double) * kSumsqBlocks) &&
              alloc((void **)&xpart, sizeof(double) * (size_t)K * kDotBlocks) &&
              alloc((void **)&xn2, sizeof(double) * K) && alloc((void **)&xf, sizeof(double) * K) && alloc((void **)&sc, sizeof(double) * 4);
    if (ok && K > 1 && !values_em) ok = alloc((void **)&vem, sizeof(float) * (size_t)nnz * K);
    int rc = ok ? CIH_OK : fail(CIH_ERR_NOMEM, "spmv: device memory");
    if (!rc) {
        if (K > 1 && !values_em) {
            count_launches(1);
            k_vals_em<<<grid_for(nnz * K), kThreads, 0, st>>>(K, nnz, val, vem);
        } else {
            vem = const_cast<float *>(val);
        }
        cudaMemsetAsync(yfix, 0, sizeof(unsigned long long) * (size_t)n, st);
        count_launches(4);
        k_upper_sumsq<<<kSumsqGrid, kSumsqThreads, 0, st>>>(RowRange{0, dim, 0}, K, rowptr, vem, partial);
        launch_dots(kSumUnit, dim, K, 1, x, n, x, xpart, xn2, nullptr, nullptr, xf, nullptr, st);
        k_mirror_scale<<<1, kSumsqBlocks, 0, st>>>(partial, K, xn2, sc);
        k_split<<<grid_for(n), kThreads, 0, st>>>(n, x, sc, xs, xm);
        launch_spmv(RowRange{0, dim, 0}, K, rowptr, col, vem, xs, xm, yrow, yfix, st);
        k_sym_finish<<<grid_for(n), kThreads, 0, st>>>(n, sc, yrow, y, yfix);
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) rc = cuda_fail(e, "spmv kernels");
    }
    for (void *p : bufs) cudaFreeAsync(p, st);
    return rc;
}


int upper_sumsq(const cih_basis &b, const int64_t *rowptr, int64_t r0, int64_t r1, const float *val, int K,
                bool values_em, double *f2, cudaStream_t st)
{
    *f2 = 0.0;
    if (r1 <= r0) return CIH_OK;
    if (K > kThreads) return fail(CIH_ERR_UNSUPPORTED, "upper_sumsq: at most 256 sets per call");
    int64_t ends[2] = {0, 0};
    cudaError_t e = cudaMemcpyAsync(&ends[0], rowptr + r0, sizeof(int64_t), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaMemcpyAsync(&ends[1], rowptr + r1, sizeof(int64_t), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return cuda_fail(e, "upper_sumsq: read nnz");
    const int64_t nnz = ends[1] - ends[0];
    float *vem = const_cast<float *>(val);
    double *partial = nullptr;
    if (cudaMallocFromPoolAsync((void **)&partial, sizeof(double) * kSumsqBlocks, b.pool, st) != cudaSuccess) {
        (void)cudaGetLastError();
        return fail(CIH_ERR_NOMEM, "upper_sumsq: device memory");
    }
    int rc = CIH_OK;
    if (K > 1 && !values_em) {
        if (cudaMallocFromPoolAsync((void **)&vem, std::max<size_t>(sizeof(float) * (size_t)nnz * K, 16), b.pool, st) !=
            cudaSuccess) {
            (void)cudaGetLastError();
            cudaFreeAsync(partial, st);
            return fail(CIH_ERR_NOMEM, "upper_sumsq: device memory");
        }
        count_launches(1);
        k_vals_em<<<grid_for(nnz * K), kThreads, 0, st>>>(K, nnz, val, vem);
    }
    count_launches(1);
    k_upper_sumsq<<<kSumsqGrid, kSumsqThreads, 0, st>>>(RowRange{r0, r1, ends[0]}, K, rowptr, vem, partial);
    std::vector<double> hp(kSumsqBlocks);
    e = cudaMemcpyAsync(hp.data(), partial, sizeof(double) * kSumsqBlocks, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) rc = cuda_fail(e, "upper_sumsq");
    for (int d = kSumsqBlocks / 2; d > 0; d >>= 1)                          // the order k_mirror_scale adds in
        for (int k = 0; k < d; ++k) hp[k] += hp[k + d];
    if (!rc) *f2 = hp[0];
    cudaFreeAsync(partial, st);
    if (vem != val) cudaFreeAsync(vem, st);
    return rc;
}

}  // namespace cih
