// Count, fill and adjoint passes over the half-stored Hamiltonian.
//
// Sec. 4.1: the nonzeros are run through twice, once to count them so the
// arrays can be allocated, once to compute them; Sec. 2: only half of the
// symmetric matrix is generated and stored; Sec. 1: every element is
// independent of the others.
//
// Row i = (proton sub-det p, neutron sub-det n).  Its stored columns j >= i,
// in ascending order:
//   A. q = p: the diagonal, then n's forward same-class neighbours inside
//      p's partner range (neutron one- and two-moves);
//   B. q > p: p's forward same-class neighbours (proton one- and two-moves)
//      and its one-move neighbours in later classes; for each q the neutron
//      partners are n itself (if it lies in q's range) merged with n's
//      one-move neighbours inside q's range (two-moves of p need n_j = n).
// The segment of n's one-move list that lies inside q's range depends on q's
// class and quanta only.  So p's one-moves are grouped by (class, N) at basis
// set-up (some 20 groups for 150 one-moves), and a warp owning a row places
// the whole row in one step: a lane per group reads the segment bounds from
// n's bucket directory, and a warp scan gives every group's place in the row.
// The count pass is the sum of the same terms.  (Walking the candidate sub-dets
// one by one, 670 a row at 4+4 Nmax=6 of which 89 % gave nothing, cost 10.9 warp
// instructions per stored nonzero: 458 us a fill at 4+4 Nmax=4 and 12.4 ms an
// adjoint at 4+4 Nmax=6, against 364 us and 8.3 ms by groups.)
//
// Matrix elements (bra = row i, ket = column j, R = orbitals common to both):
// the operator a+_a a+_b a_d a_c with a<b in the bra and c<d in the ket has
// the sign (-1)^(sum over x in {a,b,c,d} of #R below x); a one-move a <- c
// has the sign (-1)^(#R below a + #R below c) and sums V(ak, ck) over the
// spectators k in R in ascending combined order.  Proton and neutron moves
// of a pn element factorise (the cross-species counts cancel in pairs).
#include <algorithm>
#include <cmath>
#include <cstdlib>
#include <map>
#include <mutex>
#include <type_traits>

#include "cih_internal.h"
#include "ham_common.cuh"

namespace cih {
namespace {

// What the fill writes and reads: K two-body sets, table entry t of set k at
// tbme[k * tb_sk + t * tb_si] (set-major: tb_sk = table length, tb_si = 1;
// interleaved: tb_sk = 1, tb_si = K).
struct FillArgs {
    int K;
    double hw;
    const float *tbme;
    int64_t tb_sk, tb_si;
    int vec4;                 // interleaved, K % 4 == 0, 16-byte aligned: float4 table reads (and
                              // float4 value writes when em)
    int em;                   // values element-major: val[e * K + k] (else set-major val[k * nnz + e])
    const double *esp;        // combined orbital energies or null
    int32_t *col;
    float *val;               // K x nnz
    int sharded;              // 1: col / val hold only the rows from shard_row on (positions
    int64_t shard_row;        //    relative to rowptr[shard_row], nnz = that shard's count)
    const double *t1;         // one-body table (OneBodyLayout) in place of the orbital energies, or null
    float tol_one, tol_diag;  // split order (fill_splits): see near_tie
};

// The tables of up to four sets prepared for the fill (k_fill_prep), all in one
// allocation, every entry the KV values of the sets together (KV = 1, 2 or 4):
//   sq      the pn groups as full squares: no ordering of the pair indices, and
//           a proton move's entries for one neutron orbital are contiguous;
//   hi, lo  per species and forward slot: a two-move's signed value (hi); a
//           one-move's sum over its own species (one-body term, then the
//           spectators ascending) as a pair hi + lo, unsigned;
//   d       per species and sub-det: its own part of the diagonal.
// These depend on one sub-det (pair) and are used by every row that holds it:
// some 40 rows each at 4+4 Nmax=6.
struct FillWork {
    float *sq;
    float *hi[2], *lo[2];
    float2 *d[2];
    int k0, ks;               // the sets k0 .. k0 + ks - 1, ks <= KV
};

// KV values of an entry, loaded and stored together
template <int KV>
struct alignas(4 * KV) Vals {
    float v[KV];
};
// table index of t_ac for combined orbitals a, c (either order), -1 if they
// are not one group of the one-body layout
__device__ __forceinline__ int onebody_at(const DevBasis &B, int a, int c)
{
    const int g = B.ob_grp[a];
    if (g < 0 || g != B.ob_grp[c]) return -1;
    int u = B.ob_loc[a], v = B.ob_loc[c];
    if (u > v) { const int x = u; u = v; v = x; }
    const int n = B.ob_gsize[g];
    return B.ob_goff[g] + u * n - ((u * (u - 1)) >> 1) + (v - u);
}

// t_ac of a one-particle move as a double-float pair (zero without a one-body
// table); a pair outside the layout is flagged
__device__ __forceinline__ DF onebody_term(const DevBasis &B, const FillArgs &F, int a, int c, int *status)
{
    if (!F.t1) return df_of(0.f);
    const int k = onebody_at(B, a, c);
    if (k < 0) {
        atomicOr(status, 1);
        return df_of(0.f);
    }
    const double t = F.t1[k];
    const float hi = (float)t;
    return DF{hi, (float)(t - (double)hi)};
}

// The elements that a CTA of k_rows fills (row_parts): 1 the diagonal, 2 the neutron
// moves, 4 the proton moves with the neutrons kept, 8 the pn elements.
__device__ __forceinline__ int row_part()
{
    return gridDim.y == 1 ? 15 : gridDim.y == 2 ? 3 << (2 * blockIdx.y) : blockIdx.y == 0 ? 3 : 2 << blockIdx.y;
}

struct GradArgs {
    int K;
    const long long *psi;     // K x dim, psi_i * 2^61 rounded (|psi_i| < 4)
    unsigned long long *acc;  // K x tbme_len fixed point, 2^56 units
};

constexpr double kFixScale = 72057594037927936.0;   // 2^56
constexpr double kPsiScale = 2305843009213693952.0;  // 2^61

// psi_i psi_j in units of 2^-58: the high 64 bits of the 128-bit product of
// the two 2^61-scaled vectors (integer arithmetic, exact but for the floor)
__device__ __forceinline__ long long psi_prod(const long long *psi, int64_t i, int64_t j)
{
    return __mul64hi(psi[i], psi[j]);
}

// ---------------------------------------------------------------- row kernel
//
// Warps walk rows independently (next_row); a CTA shares the pn index
// tables in shared memory.  For row (p, n):
//   diagonal  - the warp sums the one-body energies and every occupied pair
//               (lanes over pairs, double-float reduction);
//   A         - n's forward same-class neighbours inside p's partner range (a
//               prefix of both lists, their counts from the directory):
//               two-moves from their table index, one-moves deferred;
//   B         - p's groups, a lane each: members x (segment + n itself) +
//               two-moves of the level, placed by a warp scan.  The pn
//               elements of all groups are then emitted flattened (lane e
//               writes element e: contiguous stores, every lane busy), pp
//               two-moves likewise, proton one-moves are deferred;
//   deferred  - one-move elements, lanes over (element, spectator) pairs and
//               a segmented double-float reduction (K sets: lanes over sets).
// Inside p's own class one- and two-moves of the protons interleave: with
// c = the first place of the level's elements minus what lower levels would
// have taken, a two-move numbered i with s one-moves before it stands at
// c + i + s (len + 1), and the one-move numbered j with t two-moves before it
// starts at c + j (len + 1) + t, len being the level's segment.

constexpr int kLaneSets = 16;     // from this many sets on, multi-term sums run with lanes over sets
// Fills of fewer than kFillSets sets of a basis that fill_splits names go through a
// working copy of the table, one, two or four sets a pass (three sets at 5+6 Nmax=4
// with a one-body table: 2.91 ms, 6.57 ms from the tables, where a one-move
// gathered ten entries per set and reduced them in a tree).  From eight sets on the row
// kernel's element-major paths write whole lines.
constexpr int kFillSets = 8;
constexpr int kTakeRuns = 4;      // runs of rows a CTA from which its warps take them from a counter (next_row)
// Rows from which one vector's adjoint takes the form of k_grad_pairs + k_grad1
// (row kernel / this form: 48,917 rows 156 / 205 us, 143,792 rows 396 / 389,
// 197,822 rows 676 / 681, 814,092 rows 2,898 / 2,319, 2.2 M rows 8,082 / 6,200)
constexpr int64_t kGradPairsMin = 1 << 19;
constexpr int kSlowCap = 64;
constexpr int kMaxA = 64;
constexpr int kPairCap = kMaxA * (kMaxA - 1) / 2;

namespace sm {
constexpr int pi = 0;                                      // uint8[kPairCap]
constexpr int pj = pi + kPairCap;                          // uint8[kPairCap]
constexpr int lg = (pj + kPairCap + 15) / 16 * 16;         // int2[kLayoutCap]: table group size, offset
constexpr int e1 = lg + kLayoutCap * 8;                    // float2[kOrbCap]: one-body energies, hi + lo
constexpr int kg = e1 + kOrbCap * 8;                       // int2[64]: pn groups (pn_k)
constexpr int warp0 = kg + 64 * 8;
// per warp
constexpr int w_seg = 0;                                   // int4[32]: pn start, divisor, first member, row place
constexpr int w_ext = w_seg + 32 * 16;                     // int2[32]: segment start | len << 16, insertion point
constexpr int w_lev = w_ext + 32 * 8;                      // int4[kLevels]: own class, per level: c, len + 1, insertion point
constexpr int w_spos = w_lev + kLevels * 16;               // int32[kSlowCap]
constexpr int w_scol = w_spos + kSlowCap * 4;              // int32[kSlowCap]
constexpr int w_scode = w_scol + kSlowCap * 4;             // uint32[kSlowCap]
constexpr int w_occ = w_scode + kSlowCap * 4;              // int16[kMaxA], then int2[32]: spectator entries
constexpr int w_size = (w_occ + kMaxA * 2 + 32 * 8 + 15) / 16 * 16;
// the pn index table pn_s (int16[n_orb_p * pn_T]) follows the per-warp areas
template <int WARPS>
constexpr int S = warp0 + WARPS * w_size;
}  // namespace sm

template <int WARPS>
inline size_t smem_bytes(int nS) { return (size_t)sm::S<WARPS> + ((size_t)nS * 2 + 15) / 16 * 16; }

template <class T>
__device__ __forceinline__ T *sptr(unsigned char *base, int off) { return reinterpret_cast<T *>(base + off); }

__device__ __forceinline__ DF warp_sum(DF v, int width)
{
    for (int d = width >> 1; d > 0; d >>= 1) {
        const DF o{__shfl_xor_sync(0xffffffffu, v.hi, d, width), __shfl_xor_sync(0xffffffffu, v.lo, d, width)};
        v = df_add(v, o);
    }
    return v;
}

// warp_sum of several sums side by side (a step of one hides the other's latency)
template <int U>
__device__ __forceinline__ void warp_sums(DF (&v)[U], int width)
{
    for (int d = width >> 1; d > 0; d >>= 1)
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const DF o{__shfl_xor_sync(0xffffffffu, v[u].hi, d, width), __shfl_xor_sync(0xffffffffu, v[u].lo, d, width)};
            v[u] = df_add(v[u], o);
        }
}

// sums(width, k) for the sets k .. k + width - 1 of K, four at a time, the last one or
// two as two: the sums of an element side by side, its table entries looked up once.
// (us, one set at a time / two / four: four sets of 3+3 Nmax=2 31.4 / 27.2 / 25.2, eight
// sets of 3+4 Nmax=3 160 / 136 / 118; two sets of 2,000 rows of 4+4 Nmax=4 39.6 / 34.4 / 39.6.)
template <bool K1, class Sums>
__device__ __forceinline__ void over_sets(int K, Sums &&sums)
{
    if (K1) {
        sums(std::integral_constant<int, 1>(), 0);
        return;
    }
    int k = 0;
    for (; k + 2 < K; k += 4) sums(std::integral_constant<int, 4>(), k);
    if (k < K) sums(std::integral_constant<int, 2>(), k);
}

// Row output view: column and value pointers at the row's first element;
// the value of set k at row position e is val[e * es + k * ks].
struct RowOut {
    int32_t *col;
    float *val;
    int64_t es, ks;
    int64_t row;
    long long psir;           // adjoint with one vector: the row's own psi (2^-61 units)
};

// one single-term element (table index, sign bit) at row-relative position e
template <int MODE, bool K1>
__device__ __forceinline__ void put_single(const DevBasis &B, const FillArgs &F, const GradArgs &Gr, const RowOut &R,
                                           int e, int64_t colj, int idx, int sgn)
{
    if (MODE == 1) {
        __stcs(R.col + e, (int32_t)colj);                         // evict-first: the walk's tables stay in L2
        if (K1) {                                                // K = 1: stride 1 in either layout
            const float v = __ldg(F.tbme + idx);
            __stcs(R.val + e, sgn ? -v : v);
        } else {
            // K sets: the value of set k goes to val[e * es + k * ks]; the sign flips bit 31
            const float *t = F.tbme + (int64_t)idx * F.tb_si;
            const int sm = sgn ? (int)0x80000000 : 0;
            if (F.em) {                                          // the K values of e are contiguous
                float *o = R.val + (int64_t)e * R.es;
                if (F.vec4) {
                    const float4 *t4 = reinterpret_cast<const float4 *>(t);
                    float4 *o4 = reinterpret_cast<float4 *>(o);
#pragma unroll 4
                    for (int k4 = 0; k4 < (F.K >> 2); ++k4) {
                        float4 v = __ldg(t4 + k4);
                        v.x = __int_as_float(__float_as_int(v.x) ^ sm);
                        v.y = __int_as_float(__float_as_int(v.y) ^ sm);
                        v.z = __int_as_float(__float_as_int(v.z) ^ sm);
                        v.w = __int_as_float(__float_as_int(v.w) ^ sm);
                        o4[k4] = v;
                    }
                } else {
                    for (int k = 0; k < F.K; ++k) o[k] = __int_as_float(__float_as_int(__ldg(t + k * F.tb_sk)) ^ sm);
                }
                return;
            }
            float *out = R.val + e;
            const int64_t vs = R.ks;
            if (F.vec4) {                                        // the K values of idx are contiguous
                const float4 *t4 = reinterpret_cast<const float4 *>(t);
#pragma unroll 4
                for (int k4 = 0; k4 < (F.K >> 2); ++k4) {
                    const float4 v = __ldg(t4 + k4);
                    float *o = out + (int64_t)(4 * k4) * vs;
                    o[0] = __int_as_float(__float_as_int(v.x) ^ sm);
                    o[vs] = __int_as_float(__float_as_int(v.y) ^ sm);
                    o[2 * vs] = __int_as_float(__float_as_int(v.z) ^ sm);
                    o[3 * vs] = __int_as_float(__float_as_int(v.w) ^ sm);
                }
            } else {
                const int64_t sk = F.tb_sk;
                int k = 0;
                for (; k + 4 <= F.K; k += 4) {                   // four independent reads in flight
                    const float v0 = __ldg(t + k * sk), v1 = __ldg(t + (k + 1) * sk);
                    const float v2 = __ldg(t + (k + 2) * sk), v3 = __ldg(t + (k + 3) * sk);
                    float *o = out + (int64_t)k * vs;
                    o[0] = __int_as_float(__float_as_int(v0) ^ sm);
                    o[vs] = __int_as_float(__float_as_int(v1) ^ sm);
                    o[2 * vs] = __int_as_float(__float_as_int(v2) ^ sm);
                    o[3 * vs] = __int_as_float(__float_as_int(v3) ^ sm);
                }
                for (; k < F.K; ++k) out[(int64_t)k * vs] = __int_as_float(__float_as_int(__ldg(t + k * sk)) ^ sm);
            }
        }
    } else if (MODE == 2) {
        for (int k = 0; k < (K1 ? 1 : Gr.K); ++k) {             // w psi_i psi_j, w = 2: 2^-57 units
            const long long q = (K1 ? __mul64hi(R.psir, Gr.psi[colj]) : psi_prod(Gr.psi + (int64_t)k * B.dim, R.row, colj)) >> 1;
            atomicAdd(Gr.acc + (int64_t)k * B.tbme_len + idx, (unsigned long long)(sgn ? -q : q));
        }
    }
}

// Element-major K-set values of up to 32 single-term elements, one per lane
// (act, table index idx, sign bit sgn, row position e), written by the whole
// warp: K/4 lanes copy one element's K values as float4s, so that a store
// instruction covers whole lines.  Needs F.em, F.vec4 and K/4 dividing 32 or
// a multiple of 32.  Columns are written by the caller.
template <int KC>
__device__ __forceinline__ void put_values_coop(const FillArgs &F, const RowOut &R, bool act, int idx, int sgn, int e)
{
    const int KK = KC > 0 ? KC : F.K;                          // KC > 0: the set count at compile time
    const int lane = threadIdx.x & 31;
    const unsigned am = __ballot_sync(0xffffffffu, act);
    if (!am) return;
    const int L = KK >> 2;                                       // float4s per element
    const int last = 31 - __clz(am);
    if (L <= 32) {
        // four rounds of P elements at a time: the four table reads are in
        // flight together before their stores
        constexpr int kB = 4;
        const int P = 32 / L, sub = lane / L, q = lane % L;
        for (int j0 = 0; j0 <= last; j0 += kB * P) {
            float4 v[kB];
            int64_t at[kB];
            bool on[kB];
#pragma unroll
            for (int u = 0; u < kB; ++u) {
                const int src = j0 + u * P + sub;
                const int jidx = __shfl_sync(0xffffffffu, idx, src & 31);
                const int je = __shfl_sync(0xffffffffu, e, src & 31);
                const int js = __shfl_sync(0xffffffffu, sgn, src & 31);
                on[u] = src < 32 && ((am >> (src & 31)) & 1);
                at[u] = (int64_t)je * R.es;
                v[u] = make_float4(0.f, 0.f, 0.f, 0.f);
                if (on[u]) {
                    const int sm = js ? (int)0x80000000 : 0;
                    v[u] = __ldg(reinterpret_cast<const float4 *>(F.tbme + (int64_t)jidx * KK) + q);
                    v[u].x = __int_as_float(__float_as_int(v[u].x) ^ sm);
                    v[u].y = __int_as_float(__float_as_int(v[u].y) ^ sm);
                    v[u].z = __int_as_float(__float_as_int(v[u].z) ^ sm);
                    v[u].w = __int_as_float(__float_as_int(v[u].w) ^ sm);
                }
            }
#pragma unroll
            for (int u = 0; u < kB; ++u)                          // evict-first: the tables stay in L2
                if (on[u]) __stcs(reinterpret_cast<float4 *>(R.val + at[u]) + q, v[u]);
        }
    } else {
        for (int j = 0; j <= last; ++j) {
            const int jidx = __shfl_sync(0xffffffffu, idx, j);
            const int je = __shfl_sync(0xffffffffu, e, j);
            const int js = __shfl_sync(0xffffffffu, sgn, j);
            if (!((am >> j) & 1)) continue;
            const int sm = js ? (int)0x80000000 : 0;
            const float4 *t4 = reinterpret_cast<const float4 *>(F.tbme + (int64_t)jidx * KK);
            float4 *o4 = reinterpret_cast<float4 *>(R.val + (int64_t)je * R.es);
            for (int q = lane; q < L; q += 32) {
                float4 v = __ldg(t4 + q);
                v.x = __int_as_float(__float_as_int(v.x) ^ sm);
                v.y = __int_as_float(__float_as_int(v.y) ^ sm);
                v.z = __int_as_float(__float_as_int(v.z) ^ sm);
                v.w = __int_as_float(__float_as_int(v.w) ^ sm);
                o4[q] = v;
            }
        }
    }
}

// lanes for one element's sum over the other species' particles (at most 32:
// with 33 particles of one species there are none of the other)
__device__ __forceinline__ int term_lanes(int Zp, int Zn)
{
    int g = 1;
    while (g < 32 && (g < Zp || g < Zn)) g <<= 1;
    return g;
}

// pair l of Z items -> (i, j), i < j
__device__ __forceinline__ void pair_of(int l, int Z, int &i, int &j)
{
    i = 0;
    while (l >= Z - 1 - i) { l -= Z - 1 - i; ++i; }
    j = i + 1 + l;
}

// One species' part of the diagonal for set k, by the whole warp: the one-body
// energies and the pairs of its Z occupied orbitals occ(i) (combined), lanes
// over both, summed as a tree.
template <class Occ>
__device__ __forceinline__ DF diag_own(const DevBasis &B, const int2 *lg, const FillArgs &F, int k, int Z, Occ occ, int *status)
{
    const int lane = threadIdx.x & 31;
    DF acc = df_of(0.f);
    for (int l = lane; l < Z * (Z - 1) / 2; l += 32) {
        int i, j, sg;
        int64_t idx;
        pair_of(l, Z, i, j);
        const int a = occ(i), c = occ(j);
        if (!tbme_at(B, lg, a, c, a, c, idx, sg)) {
            if (atomicOr(status, 1) == 0) { status[2] = a | (c << 16); status[3] = 1; }
            continue;
        }
        const float v = __ldg(F.tbme + (int64_t)k * F.tb_sk + idx * F.tb_si);
        acc = df_add(acc, df_of(sg < 0 ? -v : v));
    }
    for (int i = lane; i < Z; i += 32) {
        const int a = occ(i), k1 = F.t1 ? onebody_at(B, a, a) : -1;
        const double e = F.t1 ? (k1 >= 0 ? F.t1[k1] : 0.0) : F.esp ? F.esp[a] : F.hw * ((double)B.orbN[a] + 1.5);
        const float hi = (float)e;
        acc = df_add(acc, DF{hi, (float)(e - (double)hi)});
    }
    return warp_sum(acc, 32);
}

// k_fill1 makes the sums of several terms in another order than the row kernel: per
// species, then together.  A double-float sum of terms that do not fit its 48 bits
// depends on the order by an amount far below the FP32 result's last bit, so the
// rounded results differ only where the sum lies that close to the middle of two
// floats (near_tie) and is not exact (exact_sum).  Those sums, some in ten thousand,
// the row kernel makes again in k_fill1's order on the bases whose fills of all rows
// go through k_fill1 (SPLIT): a fill's bits do not depend on its rows, on scratch or
// on a capture.  (All of them in that order cost a quarter of the time with one
// set, 40 % with seven.)
//
// How close: with u = 2^-24 and T the sum of the terms' magnitudes below a
// df_add, its operands' low parts are at most 2 u T and its own error (two rounded
// additions, and the fast two-sum where the high parts cancel) at most 12 u^2 T, so
// an order in which no term goes through more than D additions errs by at most
// 12 D u^2 T, and two orders differ by the sum of theirs (split_tolerances); 16 instead
// of 12 also covers the rounding of T and of the test itself.

// whether a sum within tol x mag of s may round to another float (NaN: yes)
__device__ __forceinline__ bool near_tie(DF s, float mag, float tol)
{
    const float r = df_round(s), e = mag * tol;
    return !(s.hi + (s.lo + e) == r && s.hi + (s.lo - e) == r);
}

// Whether every sum of the terms, in any order, is exact: the terms are multiples of
// g = the last bit of the smallest (at least 2^-24 of it), so with T <= 2^46 g a
// partial sum's high part has a last bit of at most 2^23 g, and the low parts
// stay integers below 2^24.  (Of the sums of some seven FP32 numbers of the same
// size a few per cent are exactly half-way.)
__device__ __forceinline__ bool exact_sum(float mag, unsigned least)
{
    return mag < 1e38f && (least == 0xFFFFFFFFu || mag * 2.384185791015625e-7f <= __uint_as_float(least + 1u));
}

// Of the terms of a sum: the sum of their magnitudes, and the bits less one of the
// smallest magnitude (zeros, whose bits less one are the largest number, do not count).
struct TermSizes {
    float sum = 0.f;
    unsigned least = 0xFFFFFFFFu;
    __device__ __forceinline__ void smaller(float t) { least = min(least, (__float_as_uint(t) & 0x7FFFFFFFu) - 1u); }
    __device__ __forceinline__ void add(float t)
    {
        sum += fabsf(t);
        smaller(t);
    }
    __device__ __forceinline__ void most(float t)                // the same term of another set
    {
        sum = fmaxf(sum, fabsf(t));
        smaller(t);
    }
    __device__ __forceinline__ void over(int width)              // of the lanes of a group together
    {
        for (int d = width >> 1; d > 0; d >>= 1) {
            sum += __shfl_xor_sync(0xffffffffu, sum, d, width);
            least = min(least, __shfl_xor_sync(0xffffffffu, least, d, width));
        }
    }
};

// Which sums of a row split_row makes: the diagonal, and the one-moves (neutrons first)
// whose number's block of `per` is, modulo 31, a bit.
constexpr unsigned kSplitDiagonal = 1u << 31;
__device__ __forceinline__ unsigned split_block(int t, int per) { return 1u << (t / per % 31); }

// Sums of a row again in k_fill1's order.  The diagonal: the pn pairs, and each
// species' own part.  A one-move: its terms over the other species' particles (a lane
// each, summed as a tree) and over its own species' spectators (loaded a lane each,
// summed ascending after the one-body term).  A call of its own at the row's end, so
// that the rows without such sums keep their registers; w_occ, w_lev: the row's.
__device__ __noinline__ void split_row(const DevBasis &B, const int2 *lg, const FillArgs &F, int64_t row, unsigned which,
                                       const int16_t *w_occ, const int4 *w_lev, float *val, int64_t es, int64_t ks, int *status)
{
    const int lane = threadIdx.x & 31, nbase = B.sp[1].orb_base;
    const DevSpecies &SP = B.sp[0], &SN = B.sp[1];
    const int Zp = B.nZ[0], Zn = B.nZ[1], gsz = term_lanes(Zp, Zn), i = lane % gsz, part = row_part();
    const ProtonRec PR = B.prec[B.row_p[row]];
    const int n = (int)(row - PR.colb);
    const NeutronRec NR = B.nrec[n];
    const int cA1 = max(0, B.dir[(int64_t)n * B.dir_len + PR.dirA] - NR.self);
    int c1 = 0;                                                 // proton one-moves with n kept
    if (lane < PR.ng) {
        const int4 gr = B.grp[PR.g0 + lane];
        if ((gr.w & 0xFF) > NR.N) c1 = (unsigned)gr.x >> 16;
    }
    c1 = __reduce_add_sync(0xffffffffu, c1);
    __syncwarp();                                               // after the row's first values
    for (int k = 0; k < (which & kSplitDiagonal ? F.K : 0); ++k) {
        DF acc = df_of(0.f);
        for (int x = lane / gsz; x < Zp; x += 32 / gsz) {
            if (i >= Zn) continue;
            const int a = w_occ[x], c = w_occ[Zp + i];
            int64_t idx;
            int sg;
            if (tbme_at(B, lg, a, c, a, c, idx, sg)) {
                const float v = __ldg(F.tbme + (int64_t)k * F.tb_sk + idx * F.tb_si);
                acc = df_add(acc, df_of(sg < 0 ? -v : v));
            }
        }
        acc = warp_sum(acc, 32);
        const DF dp = diag_own(B, lg, F, k, Zp, [&](int x) { return (int)w_occ[x]; }, status);
        const DF dn = diag_own(B, lg, F, k, Zn, [&](int x) { return (int)w_occ[Zp + x]; }, status);
        if (lane == 0) val[(int64_t)k * ks] = df_round(df_add(acc, df_add(dp, dn)));
    }
    const int first = part & 2 ? 0 : cA1, last = part & 4 ? cA1 + c1 : cA1;
    int per = 32;                                               // flush_slow's
    while (per > 1 && per * (B.A - 1) > 32) per >>= 1;
    for (int t0 = first; t0 < last; t0 += 32 / gsz) {
        const int t = t0 + lane / gsz;
        const bool act = t < last && (which & split_block(t, per)), neu = t < cA1;
        if (!__any_sync(0xffffffffu, act)) continue;
        int e = 0, code = 0;
        if (act && neu) {
            const int64_t sl = NR.fw + NR.fwlen - 1 - t;
            e = 1 + t + (SN.fw_rec[sl].y & 0xFFFFFF);
            code = ~SN.fw_tb[sl];
        } else if (act) {
            const int64_t sl = PR.fw + PR.fwlen - 1 - (t - cA1);
            const int o = SP.fw_rec[sl].y;
            const int4 lv = w_lev[o >> 24];
            e = lv.x + (t - cA1) * lv.y + (o & 0xFFFFFF) + lv.z;
            code = ~SP.fw_tb[sl];
        }
        const int base = neu ? nbase : 0, a = base + (code & 0xFF), c = base + ((code >> 8) & 0xFF);
        const int own0 = neu ? Zp : 0, nown = (neu ? Zn : Zp) - 1, oth0 = neu ? 0 : Zp, noth = neu ? Zp : Zn;
        int ia = 0;                                             // a's place among its species
        for (int x = 0; x <= nown; ++x) ia += (w_occ[own0 + x] < a);
        const bool ho = act && i < noth, hs = act && i < nown;
        const int ko = ho ? w_occ[oth0 + i] : 0, kx = hs ? w_occ[own0 + i + (i >= ia ? 1 : 0)] : 0;
        int64_t xo = 0, xs = 0;
        int go = 1, gs = 1;
        const bool oko = ho && tbme_at(B, lg, a, ko, c, ko, xo, go), oks = hs && tbme_at(B, lg, a, kx, c, kx, xs, gs);
        const DF one = act ? onebody_term(B, F, a, c, status) : df_of(0.f);
        for (int k = 0; k < F.K; ++k) {
            const float *tk = F.tbme + (int64_t)k * F.tb_sk;
            float to = oko ? __ldg(tk + xo * F.tb_si) : 0.f, ts = oks ? __ldg(tk + xs * F.tb_si) : 0.f;
            if (go < 0) to = -to;
            if (gs < 0) ts = -ts;
            const DF v = warp_sum(df_of(to), gsz);
            DF own = one;
            for (int x = 0; x < gsz; ++x) {
                const float y = __shfl_sync(0xffffffffu, ts, x, gsz);
                if (x < nown) own = df_add(own, df_of(y));
            }
            if (act && i == 0) {
                const float r = df_round(df_add(v, own));
                val[(int64_t)e * es + (int64_t)k * ks] = (code >> 16) & 1 ? -r : r;
            }
        }
    }
}

// Deferred one-move elements of a row: lanes over (element, spectator)
// pairs, groups of the next power of two >= A-1 lanes, segmented sum (from
// kLaneSets sets on: one element at a time, lanes over sets).
// The queue holds row-relative positions, columns and packed moves
// (bra-only a, ket-only c, sign, neutron flag in bit 31).
template <int MODE, bool K1, int EM, bool SPLIT>
__device__ __forceinline__ void flush_slow(const DevBasis &B, const int2 *lg, const FillArgs &F, const GradArgs &Gr,
                                           int *status, const int16_t *w_occ, const int32_t *w_spos,
                                           const int32_t *w_scol, const uint32_t *w_scode, int &nslow,
                                           const RowOut &R, int &flushed, unsigned &again)
{
    const int lane = threadIdx.x & 31;
    const int A = B.A, nbase = B.sp[1].orb_base;
    __syncwarp();
    const int ns = nslow;
    const int sp_n = A - 1;
    if (MODE == 1 && !K1 && (EM > 1 || F.K >= kLaneSets)) {      // (EM > 1: 64 sets)
        // K sets: the table entries of 32 / (A - 1) elements at a time (lanes
        // over (element, spectator) pairs, so their lookups run together), then
        // per element lanes over sets sum them in spectator order
        int2 *spec = reinterpret_cast<int2 *>(const_cast<int16_t *>(w_occ) + kMaxA);
        const int per = sp_n > 0 ? 32 / sp_n : 32;
        for (int e0 = 0; e0 < ns; e0 += per) {
            {
                const int ei = sp_n > 0 ? lane / sp_n : lane, i = sp_n > 0 ? lane % sp_n : 0;
                const int e = e0 + ei;
                if (ei < per && e < ns && i < sp_n) {
                    const uint32_t code = w_scode[e];
                    const int base = (code >> 31) ? nbase : 0;
                    const int a = base + (int)(code & 0xFF), c = base + (int)((code >> 8) & 0xFF);
                    int ia = 0;
                    for (int x = 0; x < A; ++x) ia += (w_occ[x] < a);
                    const int kspec = w_occ[i + (i >= ia ? 1 : 0)];
                    int64_t idx = 0;
                    int sg = 1;
                    const bool ok = tbme_at(B, lg, a, kspec, c, kspec, idx, sg);
                    if (!ok && atomicOr(status, 1) == 0) {
                        status[2] = a | (c << 16);
                        status[3] = 2 | (kspec << 8);
                    }
                    spec[ei * sp_n + i] = make_int2(ok ? (int)idx : -1, sg);
                }
            }
            __syncwarp();
            const int ne = min(per, ns - e0);
            const int KK = EM > 1 ? EM : F.K;                 // EM > 1: the set count at compile time
            const int L4 = KK >> 2;
            if (EM) {
                // element-major values: K/4 lanes per element with float4 reads and
                // writes, 32 / (K/4) elements at a time; each set's sum in the same
                // order as below
                const int P = 32 / L4, sub = lane / L4, q4 = lane % L4;
                for (int j0 = 0; j0 < ne; j0 += P) {
                    const int j = j0 + sub;
                    if (j >= ne) continue;
                    const int e = e0 + j;
                    const uint32_t code = w_scode[e];
                    const int base = (code >> 31) ? nbase : 0;
                    const int a = base + (int)(code & 0xFF), c = base + (int)((code >> 8) & 0xFF);
                    const int sgn = (code >> 16) & 1;
                    const int eo = w_spos[e];
                    const DF t1v = onebody_term(B, F, a, c, status);
                    const int2 *sj = spec + j * sp_n;
                    DF v0 = t1v, v1 = t1v, v2 = t1v, v3 = t1v;
#pragma unroll 8
                    for (int i = 0; i < sp_n; ++i) {
                        const int2 q = sj[i];
                        if (q.x < 0) continue;
                        float4 t = __ldg(reinterpret_cast<const float4 *>(F.tbme + (int64_t)q.x * KK) + q4);
                        if (q.y < 0) { t.x = -t.x; t.y = -t.y; t.z = -t.z; t.w = -t.w; }
                        v0 = df_add(v0, df_of(t.x));
                        v1 = df_add(v1, df_of(t.y));
                        v2 = df_add(v2, df_of(t.z));
                        v3 = df_add(v3, df_of(t.w));
                    }
                    float4 r = make_float4(df_round(v0), df_round(v1), df_round(v2), df_round(v3));
                    if (sgn) { r.x = -r.x; r.y = -r.y; r.z = -r.z; r.w = -r.w; }
                    __stcs(reinterpret_cast<float4 *>(R.val + (int64_t)eo * R.es) + q4, r);
                    if (q4 == 0) R.col[eo] = w_scol[e];
                }
            }
            for (int j = 0; j < (EM ? 0 : ne); ++j) {                // the other layouts: one element at a time
                const int e = e0 + j;
                const uint32_t code = w_scode[e];
                const int base = (code >> 31) ? nbase : 0;
                const int a = base + (int)(code & 0xFF), c = base + (int)((code >> 8) & 0xFF);
                const int sgn = (code >> 16) & 1;
                const int eo = w_spos[e];
                const DF t1v = onebody_term(B, F, a, c, status);      // the one-body term first
                const int2 *sj = spec + j * sp_n;
                for (int k = lane; k < F.K; k += 32) {
                    DF v = t1v;
#pragma unroll 8
                    for (int i = 0; i < sp_n; ++i) {
                        const int2 q = sj[i];
                        if (q.x < 0) continue;
                        const float t = __ldg(F.tbme + (int64_t)k * F.tb_sk + (int64_t)q.x * F.tb_si);
                        v = df_add(v, df_of(q.y < 0 ? -t : t));
                    }
                    const float r = df_round(v);
                    R.val[(int64_t)eo * R.es + (int64_t)k * R.ks] = sgn ? -r : r;
                }
                if (lane == 0) R.col[eo] = w_scol[e];
            }
            __syncwarp();
        }
        nslow = 0;
        return;
    }
    int gsz = 1;
    while (gsz < sp_n) gsz <<= 1;
    const int per = 32 / gsz;
    for (int e0 = 0; EM <= 1 && e0 < ns; e0 += per) {
        const int e = e0 + lane / gsz;
        const int i = lane % gsz;
        const bool act = e < ns;
        const uint32_t code = act ? w_scode[e] : 0;
        const int base = (code >> 31) ? nbase : 0;
        const int a = base + (int)(code & 0xFF), c = base + (int)((code >> 8) & 0xFF);
        const int sgn = (code >> 16) & 1;
        int ia = 0;
        for (int x = 0; x < A; ++x) ia += (w_occ[x] < a);
        const bool has = act && i < sp_n;
        const int kspec = has ? w_occ[i + (i >= ia ? 1 : 0)] : 0;
        const int eo = act ? w_spos[e] : 0;
        const int64_t colj = act ? w_scol[e] : 0;
        int64_t idx = 0;
        int sg = 1;
        bool ok = true;
        if (has) ok = tbme_at(B, lg, a, kspec, c, kspec, idx, sg);
        if (!ok && atomicOr(status, 1) == 0) {
            status[2] = a | (c << 16);
            status[3] = 2 | (kspec << 8);
        }
        // the one-body term t_ac (one per element: added by its group's first lane)
        const DF t1v = (MODE == 1 && act && i == 0) ? onebody_term(B, F, a, c, status) : df_of(0.f);
        if (MODE == 1) {
            TermSizes z;                                        // SPLIT: of the lane's terms, all sets together
            bool near = false;
            auto sums = [&](auto width, int k0) {               // the sets from k0 on
                constexpr int U = decltype(width)::value;
                DF v[U];
                unsigned most = 0;
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    float t = 0.f;
                    if (has && ok && (K1 || k0 + u < F.K)) t = __ldg(F.tbme + (int64_t)(k0 + u) * F.tb_sk + idx * F.tb_si);
                    if (SPLIT) {
                        z.most(t);
                        most = max(most, __float_as_uint(t) & 0x7FFFFFFFu);
                    }
                    v[u] = df_of(sg < 0 ? -t : t);
                }
#pragma unroll
                for (int u = 0; u < U; ++u) v[u] = df_add(t1v, v[u]);
                warp_sums<U>(v, gsz);
                if (SPLIT) {
                    const float mag = fabsf(t1v.hi) + __uint_as_float(__reduce_max_sync(0xffffffffu, most)) * (float)sp_n;
#pragma unroll
                    for (int u = 0; u < U; ++u) near |= (K1 || k0 + u < F.K) && near_tie(v[u], mag, F.tol_one);
                }
                if (act && i == 0) {
                    if (k0 == 0) R.col[eo] = (int32_t)colj;
#pragma unroll
                    for (int u = 0; u < U; ++u) {
                        const float r = df_round(v[u]);
                        if (K1 || k0 + u < F.K) R.val[(int64_t)eo * R.es + (int64_t)(k0 + u) * R.ks] = sgn ? -r : r;
                    }
                }
            };
            over_sets<K1>(K1 ? 1 : F.K, sums);
            near = near && act && i == 0;
            if (SPLIT && __any_sync(0xffffffffu, near)) {
                z.add(t1v.hi);
                z.add(t1v.lo);
                z.over(gsz);
                if (near && !exact_sum(z.sum, z.least)) again |= split_block(flushed + e, per);
            }
        } else if (has && ok) {
            for (int kk = 0; kk < (K1 ? 1 : Gr.K); ++kk) {
                const long long q =
                    (K1 ? __mul64hi(R.psir, Gr.psi[colj]) : psi_prod(Gr.psi + (int64_t)kk * B.dim, R.row, colj)) >> 1;
                const bool neg = (sgn != 0) != (sg < 0);
                atomicAdd(Gr.acc + (int64_t)kk * B.tbme_len + idx, (unsigned long long)(neg ? -q : q));
            }
        }
    }
    __syncwarp();
    if (SPLIT) flushed += ns;
    nslow = 0;
}

// The rows of a CTA are the runs of WARPS rows blockIdx.x, blockIdx.x + gridDim.x,
// ... of its range; its warps take them one by one, the first run without asking,
// the rest from a counter in shared memory (WARPS before the first call).  Rows differ
// in length, and a warp's rows, at fixed distances, alike: with every warp taking its
// own, the longest warp had 1.8 times the mean at 3+4 Nmax=4 (11 rows each), 1.4 at
// 4+4 Nmax=4, 1.1 at 4+4 Nmax=6.  us, own rows / taken: one-set fill 132 / 119, 306 /
// 290, 5,770 / 5,610 there; adjoint at 4+4 Nmax=4 375 / 344; 64 sets at 3+4 Nmax=4 849 /
// 668.  Up to kTakeRuns runs the counter costs what it gains (5+5 Nmax=2, 14,502 rows,
// eight sets: 199 / 207).
template <int WARPS>
__device__ __forceinline__ int64_t first_row(int64_t r0, int wid) { return r0 + (int64_t)blockIdx.x * WARPS + wid; }

template <int WARPS>
__device__ __forceinline__ int64_t next_row(int64_t row, int64_t r0, int64_t r1, int *counter, int lane)
{
    const int64_t run = (int64_t)gridDim.x * WARPS;             // rows of one run of every CTA
    if (r1 - r0 <= kTakeRuns * run) return row + run;
    int t = lane == 0 ? atomicAdd(counter, 1) : 0;
    t = __shfl_sync(0xffffffffu, t, 0);
    return r0 + (t / WARPS) * run + (int64_t)blockIdx.x * WARPS + t % WARPS;
}

template <int MODE, bool K1, int WARPS, int EM, bool SPLIT>
__device__ __forceinline__ void walk_rows(const DevBasis &B, const int64_t *rowptr, int64_t *counts, const FillArgs &F, const GradArgs &Gr,
                                          int64_t r0, int64_t r1, int *status)
{
    constexpr int kThreads = WARPS * 32;
    extern __shared__ __align__(16) unsigned char sb[];
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const unsigned lt = (1u << lane) - 1;
    const DevSpecies &SP = B.sp[0], &SN = B.sp[1];
    const int A = B.A, nbase = SN.orb_base;
    const int npairs = A * (A - 1) / 2;
    const int T = B.pn_T;
    int2 *KG = sptr<int2>(sb, sm::kg);
    int16_t *XS = sptr<int16_t>(sb, sm::S<WARPS>);
    __shared__ int taken;
    if (tid == 0) taken = WARPS;
    if (MODE == 0) __syncthreads();
    if (MODE != 0) {
        for (int i = tid; i < SP.n_orb * T; i += kThreads) XS[i] = B.pn_s[i];
        for (int i = tid; i < 64; i += kThreads) KG[i] = B.pn_k[i];
        if (B.ngroups <= kLayoutCap) {
            int2 *lgw = sptr<int2>(sb, sm::lg);
            for (int g = tid; g < B.ngroups; g += kThreads) lgw[g] = make_int2(B.gsize[g], (int)B.goff[g]);
        }
        if (MODE == 1) {                                   // one-body energies as hi + lo pairs
            float2 *e1w = sptr<float2>(sb, sm::e1);
            for (int a = tid; a < B.ntot && a < kOrbCap; a += kThreads) {
                const int k1 = F.t1 ? onebody_at(B, a, a) : -1;
                const double e = F.t1 ? (k1 >= 0 ? F.t1[k1] : 0.0) : F.esp ? F.esp[a] : F.hw * ((double)B.orbN[a] + 1.5);
                const float hi = (float)e;
                e1w[a] = make_float2(hi, (float)(e - (double)hi));
            }
        }
        uint8_t *pi = sptr<uint8_t>(sb, sm::pi), *pj = sptr<uint8_t>(sb, sm::pj);
        for (int l = tid; l < npairs; l += kThreads) {     // pair l -> (i, j), i < j
            int i = 0, r = l;
            while (r >= A - 1 - i) { r -= A - 1 - i; ++i; }
            pi[l] = (uint8_t)i;
            pj[l] = (uint8_t)(i + 1 + r);
        }
        __syncthreads();
    }
    // stored nonzeros the output arrays hold, and the row pointer of their first element
    const int64_t sbase = (MODE == 1 && F.sharded) ? rowptr[F.shard_row] : 0;
    const int64_t nnz = MODE == 1 ? (F.sharded ? rowptr[r1] - sbase : rowptr[B.dim]) : 0;
    const int2 *lg = sptr<int2>(sb, sm::lg);
    unsigned char *wb = sb + sm::warp0 + wid * sm::w_size;
    int4 *w_seg = sptr<int4>(wb, sm::w_seg), *w_lev = sptr<int4>(wb, sm::w_lev);
    int2 *w_ext = sptr<int2>(wb, sm::w_ext);
    int32_t *w_spos = sptr<int32_t>(wb, sm::w_spos), *w_scol = sptr<int32_t>(wb, sm::w_scol);
    uint32_t *w_scode = sptr<uint32_t>(wb, sm::w_scode);
    int16_t *w_occ = sptr<int16_t>(wb, sm::w_occ);
    const int Zpro = B.nZ[0], Zneu = B.nZ[1];
    // K sets, element-major values: warp-cooperative value writes
    // (EM: the launcher chose this instantiation because F.em, F.vec4 and
    // K/4 dividing 32 or a multiple of 32 hold; the other K-set layouts
    // compile without these paths, and these without theirs)
    constexpr bool coop = MODE == 1 && !K1 && EM;

    for (int64_t row = first_row<WARPS>(r0, wid); row < r1; row = next_row<WARPS>(row, r0, r1, &taken, lane)) {
        const int p = B.row_p[row];
        const ProtonRec PR = B.prec[p];
        const int n = (int)(row - PR.colb);
        const NeutronRec NR = B.nrec[n];
        RowOut R;
        R.row = row;
        R.psir = (MODE == 2 && K1) ? Gr.psi[row] : 0;
        R.es = (MODE == 1 && F.em) ? (EM > 1 ? EM : F.K) : 1;
        R.ks = (MODE == 1 && F.em) ? 1 : nnz;
        int rowlen = 0;
        if (MODE == 1) {
            const int64_t r0 = rowptr[row] - sbase;
            rowlen = (int)(min(rowptr[row + 1] - sbase, nnz) - r0);
            R.col = F.col + r0;
            R.val = F.val + r0 * R.es;
        }
        int nslow = 0;
        unsigned again = 0;                                     // SPLIT: sums of the row that may depend on the order

        // ---- diagonal: occupied orbitals (combined, ascending), then all pairs
        if (MODE != 0) {
            for (int i = lane; i < A; i += 32)
                w_occ[i] = i < Zpro ? (int16_t)B.occ[0][(int64_t)p * Zpro + i]
                                    : (int16_t)(nbase + B.occ[1][(int64_t)n * Zneu + (i - Zpro)]);
            __syncwarp();
        }
        if (MODE == 2 || (MODE == 1 && (row_part() & 1))) {
            const uint8_t *pi = sptr<uint8_t>(sb, sm::pi), *pj = sptr<uint8_t>(sb, sm::pj);
            const bool kset = MODE == 1 && !K1 && F.K >= kLaneSets && npairs <= kSlowCap;
            if (kset) {
                // K sets: the pairs' table entries in the (still empty) deferred
                // queue arrays, then lanes over sets sum them in pair order
                for (int l = lane; l < npairs; l += 32) {
                    const int a = w_occ[pi[l]], c = w_occ[pj[l]];
                    int64_t idx;
                    int sg;
                    const bool ok = tbme_at(B, lg, a, c, a, c, idx, sg);
                    if (!ok && atomicOr(status, 1) == 0) { status[2] = a | (c << 16); status[3] = 1; }
                    w_scol[l] = ok ? (int32_t)idx : -1;
                    w_scode[l] = sg < 0 ? 1u : 0u;
                }
                __syncwarp();
                DF one = df_of(0.f);
                const float2 *e1 = sptr<float2>(sb, sm::e1);
                for (int i = 0; i < A; ++i) {
                    const float2 q = e1[w_occ[i]];
                    one = df_add(one, DF{q.x, q.y});
                }
                const int KK = EM > 1 ? EM : F.K;
                const int L4 = KK >> 2;
                if (EM && L4 <= 32) {
                    // element-major values: four sets per lane, float4 reads, the same
                    // per-set order as below
                    for (int q4 = lane; q4 < L4; q4 += 32) {
                        DF a0 = df_of(0.f), a1 = a0, a2 = a0, a3 = a0;
#pragma unroll 4
                        for (int l = 0; l < npairs; ++l) {
                            const int32_t idx = w_scol[l];
                            if (idx < 0) continue;
                            float4 t = __ldg(reinterpret_cast<const float4 *>(F.tbme + (int64_t)idx * KK) + q4);
                            if (w_scode[l]) { t.x = -t.x; t.y = -t.y; t.z = -t.z; t.w = -t.w; }
                            a0 = df_add(a0, df_of(t.x));
                            a1 = df_add(a1, df_of(t.y));
                            a2 = df_add(a2, df_of(t.z));
                            a3 = df_add(a3, df_of(t.w));
                        }
                        if (rowlen > 0)
                            __stcs(reinterpret_cast<float4 *>(R.val) + q4,
                                   make_float4(df_round(df_add(a0, one)), df_round(df_add(a1, one)),
                                               df_round(df_add(a2, one)), df_round(df_add(a3, one))));
                    }
                }
                for (int k = lane; k < (EM && L4 <= 32 ? 0 : F.K); k += 32) {
                    DF acc = df_of(0.f);
#pragma unroll 4
                    for (int l = 0; l < npairs; ++l) {
                        const int32_t idx = w_scol[l];
                        if (idx < 0) continue;
                        const float v = __ldg(F.tbme + (int64_t)k * F.tb_sk + (int64_t)idx * F.tb_si);
                        acc = df_add(acc, df_of(w_scode[l] ? -v : v));
                    }
                    if (rowlen > 0) R.val[(int64_t)k * R.ks] = df_round(df_add(acc, one));
                }
                if (lane == 0 && rowlen > 0) R.col[0] = (int32_t)row;
                __syncwarp();
            }
            auto sums = [&](auto width, int k0) {               // the sets from k0 on
                constexpr int U = decltype(width)::value;
                DF acc[U];
                TermSizes z;
#pragma unroll
                for (int u = 0; u < U; ++u) acc[u] = df_of(0.f);
                for (int l = lane; l < npairs; l += 32) {
                    const int a = w_occ[pi[l]], c = w_occ[pj[l]];
                    int64_t idx;
                    int sg;
                    if (!tbme_at(B, lg, a, c, a, c, idx, sg)) {
                        if (atomicOr(status, 1) == 0) { status[2] = a | (c << 16); status[3] = 1; }
                        continue;
                    }
                    float m = 0.f;
#pragma unroll
                    for (int u = 0; u < U; ++u) {
                        const float v = K1 || k0 + u < F.K ? __ldg(F.tbme + (int64_t)(k0 + u) * F.tb_sk + idx * F.tb_si) : 0.f;
                        acc[u] = df_add(acc[u], df_of(sg < 0 ? -v : v));
                        if (SPLIT) {
                            m = fmaxf(m, fabsf(v));
                            z.smaller(v);
                        }
                    }
                    if (SPLIT) z.sum += m;
                }
                const float2 *e1 = sptr<float2>(sb, sm::e1);
                for (int i = lane; i < A; i += 32) {
                    const float2 q = e1[w_occ[i]];
#pragma unroll
                    for (int u = 0; u < U; ++u) acc[u] = df_add(acc[u], DF{q.x, q.y});
                    if (SPLIT) {
                        z.add(q.x);
                        z.add(q.y);
                    }
                }
                warp_sums<U>(acc, 32);
                if (lane == 0 && rowlen > 0) {
                    if (k0 == 0) R.col[0] = (int32_t)row;
#pragma unroll
                    for (int u = 0; u < U; ++u)
                        if (K1 || k0 + u < F.K) R.val[(int64_t)(k0 + u) * R.ks] = df_round(acc[u]);
                }
                if (SPLIT) {
                    const float mag = 32.f * __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(z.sum)));
                    bool near = false;
#pragma unroll
                    for (int u = 0; u < U; ++u) near |= (K1 || k0 + u < F.K) && near_tie(acc[u], mag, F.tol_diag);
                    if (__any_sync(0xffffffffu, near)) {      // look closer
                        z.over(32);
#pragma unroll
                        for (int u = 0; u < U; ++u)
                            if ((K1 || k0 + u < F.K) && near_tie(acc[u], z.sum, F.tol_diag) && !exact_sum(z.sum, z.least))
                                again |= kSplitDiagonal;
                    }
                }
            };
            if constexpr (MODE == 2) {
                for (int k = 0; k < (K1 ? 1 : Gr.K); ++k) {
                    for (int l = lane; l < npairs; l += 32) {
                        const int a = w_occ[pi[l]], c = w_occ[pj[l]];
                        int64_t idx;
                        int sg;
                        if (!tbme_at(B, lg, a, c, a, c, idx, sg)) {
                            if (atomicOr(status, 1) == 0) { status[2] = a | (c << 16); status[3] = 1; }
                            continue;
                        }
                        const long long q = psi_prod(Gr.psi + (int64_t)k * B.dim, row, row) >> 2;    // w = 1 on the diagonal
                        atomicAdd(Gr.acc + (int64_t)k * B.tbme_len + idx, (unsigned long long)(sg < 0 ? -q : q));
                    }
                }
            } else if (!kset) {
                over_sets<K1>(K1 ? 1 : F.K, sums);
            }
        }

        // ---- A: same-class forward neutron neighbours inside p's range
        const int16_t *dirn = B.dir + (int64_t)n * B.dir_len;
        const int cA1 = max(0, dirn[PR.dirA] - NR.self), cA2 = SN.fw_lev[(int64_t)n * SN.NL + PR.levA];
        int pos = 1 + cA1 + cA2, flushed = SPLIT && !(row_part() & 2) ? cA1 : 0;           // one-moves done (split_row's numbers)
        if (MODE == 1 && pos > rowlen) {
            if (lane == 0) atomicOr(status, 2);
            continue;
        }
        if (MODE == 2 || (MODE == 1 && (row_part() & 2))) {
            const int2 *rec = SN.fw_rec + NR.fw;
            const int32_t *tbl = SN.fw_tb + NR.fw;
            for (int t0 = 0; t0 < cA2; t0 += 32) {
                const int t = t0 + lane;
                const bool in = t < cA2;
                const int2 rc = in ? rec[t] : make_int2(0, 0);
                const int tb = in ? tbl[t] : 0;
                const int e = 1 + t + (rc.y & 0xFFFFFF);
                if (MODE == 1 && coop) {
                    if (in) __stcs(R.col + e, PR.colb + rc.x);
                    put_values_coop<(EM > 1 ? EM : 0)>(F, R, in, tb >> 1, tb & 1, e);
                } else if (in) {
                    put_single<MODE, K1>(B, F, Gr, R, e, (int64_t)(PR.colb + rc.x), tb >> 1, tb & 1);
                }
            }
            for (int t0 = 0; t0 < cA1; t0 += 32) {
                const int t = t0 + lane, c = min(32, cA1 - t0);
                if (nslow + c > kSlowCap)
                    flush_slow<MODE, K1, EM, SPLIT>(B, lg, F, Gr, status, w_occ, w_spos, w_scol, w_scode, nslow, R, flushed, again);
                if (lane < c) {
                    const int sl = NR.fwlen - 1 - t;
                    const int2 rc = rec[sl];
                    w_spos[nslow + lane] = 1 + t + (rc.y & 0xFFFFFF);
                    w_scol[nslow + lane] = PR.colb + rc.x;
                    w_scode[nslow + lane] = (uint32_t)~tbl[sl] | (1u << 31);            // neutron one-move
                }
                nslow += c;
            }
        }

        // ---- B: p's groups, a lane each
        const int2 *n1row = B.n1p + NR.n1;
        const int2 *l1row = B.l1 + PR.l1;
        const int2 *recp = SP.fw_rec + PR.fw;
        for (int g0 = 0; g0 < PR.ng; g0 += 32) {
            int4 gr = make_int4(0, 0, 0, 0);
            if (g0 + lane < PR.ng) gr = B.grp[PR.g0 + g0 + lane];
            const int n1c = (unsigned)gr.x >> 16, s0 = dirn[gr.y & 0xFFFF], len = dirn[(unsigned)gr.y >> 16] - s0;
            const int self = (gr.w & 0xFF) > NR.N ? 1 : 0;                  // own class and N_n <= L_q
            const int npn = n1c * len, tot = npn + self * (n1c + gr.z);
            if (MODE == 0) {
                pos += __reduce_add_sync(0xffffffffu, tot);
                continue;
            }
            int itot = tot, ipn = npn;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const int o1 = __shfl_up_sync(0xffffffffu, itot, d), o2 = __shfl_up_sync(0xffffffffu, ipn, d);
                if (lane >= d) { itot += o1; ipn += o2; }
            }
            const int Tall = __shfl_sync(0xffffffffu, itot, 31), Tpn = __shfl_sync(0xffffffffu, ipn, 31);
            if (MODE == 1 && pos + Tall > rowlen) {
                if (lane == 0) atomicOr(status, 2);
                rowlen = -1;                                    // (no second look at an incomplete row)
                break;
            }
            const int at0 = pos + itot - tot, st = ipn - npn, f1 = gr.x & 0xFFFF;
            const int ins = NR.self - s0;                                   // where n sorts in the segment
            const int c = at0 - f1 * (len + 1) - (gr.w >> 8);
            const unsigned ne = __ballot_sync(0xffffffffu, npn > 0);
            if (npn > 0) {
                const int j = __popc(ne & lt);
                w_seg[j] = make_int4(st, (int)(0xFFFFFFFFu / (unsigned)len), f1, self ? c : at0 - st);
                w_ext[j] = make_int2(s0 | len << 16, self ? ins : -1);
            }
            int c1 = 0, c2 = 0;
            if (g0 == 0) {                                      // own-class groups come first, at most 32
                if (gr.w) w_lev[((B.Nlim - (gr.w & 0xFF) + 1) - SP.N0) >> 1] = make_int4(c, len + 1, ins, 0);
                c1 = MODE == 2 || (row_part() & 4) ? __reduce_add_sync(0xffffffffu, self * n1c) : 0;
                c2 = MODE == 2 || (row_part() & 4) ? __reduce_add_sync(0xffffffffu, self * gr.z) : 0;
            }
            __syncwarp();
            // pp two-moves: a prefix of p's list
            for (int t0 = 0; t0 < c2; t0 += 32) {
                const int t = t0 + lane;
                const bool in = t < c2;
                int e = 0, col = 0, tb = 0;
                if (in) {
                    const int2 rc = recp[t];
                    const int4 lv = w_lev[rc.y >> 24];
                    tb = SP.fw_tb[PR.fw + t];
                    e = lv.x + t + (rc.y & 0xFFFFFF) * lv.y;
                    col = rc.x + n;
                }
                if (MODE == 1 && coop) {
                    if (in) __stcs(R.col + e, col);
                    put_values_coop<(EM > 1 ? EM : 0)>(F, R, in, tb >> 1, tb & 1, e);
                } else if (in) {
                    put_single<MODE, K1>(B, F, Gr, R, e, (int64_t)col, tb >> 1, tb & 1);
                }
            }
            // proton one-moves with n kept: a prefix of p's one-moves
            for (int t0 = 0; t0 < c1; t0 += 32) {
                const int t = t0 + lane, cc = min(32, c1 - t0);
                if (nslow + cc > kSlowCap)
                    flush_slow<MODE, K1, EM, SPLIT>(B, lg, F, Gr, status, w_occ, w_spos, w_scol, w_scode, nslow, R, flushed, again);
                if (lane < cc) {
                    const int2 q = l1row[t];
                    const int o = recp[PR.fwlen - 1 - t].y;
                    const int4 lv = w_lev[o >> 24];
                    w_spos[nslow + lane] = lv.x + t * lv.y + (o & 0xFFFFFF) + lv.z;
                    w_scol[nslow + lane] = q.x + n;
                    w_scode[nslow + lane] = (uint32_t)q.y;
                }
                nslow += cc;
            }
            // pn elements of all groups, flattened: element e belongs to the last
            // non-empty group starting at or before e.  Per 32-element window, a
            // mask of the group starts inside it (OR over lanes) and the count of
            // earlier starts give the group; the member and the place in its
            // segment are the quotient and remainder by the segment length.
            const unsigned le = (2u << lane) - 1u;                 // bits 0..lane
            int before = 0;                                        // groups started before the window
            for (int w0 = MODE == 2 || (row_part() & 8) ? 0 : Tpn; w0 < Tpn; w0 += 32) {
                const unsigned mk = __reduce_or_sync(0xffffffffu, npn > 0 && st >= w0 && st < w0 + 32 ? 1u << (st - w0) : 0u);
                const int e = w0 + lane;
                int at = 0, idx = 0, sg = 0;
                if (e < Tpn) {
                    const int j = before + __popc(mk & le) - 1;
                    const int4 sg4 = w_seg[j];
                    const int2 sx = w_ext[j];
                    const int rel = e - sg4.x, ln = (unsigned)sx.x >> 16;
                    int qi = (int)__umulhi((unsigned)rel, (unsigned)sg4.y), k = rel - qi * ln;   // at most one short
                    if (k >= ln) { ++qi; k -= ln; }
                    const int i1 = sg4.z + qi;
                    const int2 q = l1row[i1], ent = n1row[(sx.x & 0xFFFF) + k];
                    at = sg4.w + e;
                    if (sx.y >= 0)                                 // n itself is among the partners
                        at = sg4.w + i1 * (ln + 1) + (recp[PR.fwlen - 1 - i1].y & 0xFFFFFF) + k + (k >= sx.y ? 1 : 0);
                    idx = pn_index_at(KG, XS, T, q.y, ent.y, sg);
                    if (MODE == 1 && coop) __stcs(R.col + at, q.x + ent.x);
                    else put_single<MODE, K1>(B, F, Gr, R, at, (int64_t)(q.x + ent.x), idx, sg);
                }
                if (MODE == 1 && coop) put_values_coop<(EM > 1 ? EM : 0)>(F, R, e < Tpn, idx, sg, at);
                before += __popc(mk);
            }
            __syncwarp();
            pos += Tall;
        }
        if (MODE != 0 && nslow > 0) flush_slow<MODE, K1, EM, SPLIT>(B, lg, F, Gr, status, w_occ, w_spos, w_scol, w_scode, nslow, R, flushed, again);
        if (SPLIT) {
            again = __reduce_or_sync(0xffffffffu, rowlen > 0 ? again : 0);
            if (again) split_row(B, lg, F, row, again, w_occ, w_lev, R.val, R.es, R.ks, status);
        }
        if (MODE == 0 && lane == 0) counts[row] = pos;
        __syncwarp();
    }
}

// Two forms of the same kernel: with grid-constant parameters ptxas spills less for one
// set (20 bytes against 24, 36 against 40 with SPLIT), but the loops over sets run slower
// (64 sets of 3+4 Nmax=3, set-major: 780 us against 646).
template <int MODE, bool K1, int WARPS, int EM, bool SPLIT = false>
__global__ void __launch_bounds__(WARPS * 32, 32 / WARPS)
k_rows(DevBasis B, const int64_t *rowptr, int64_t *counts, FillArgs F, GradArgs Gr, int64_t r0, int64_t r1, int *status)
{
    walk_rows<MODE, K1, WARPS, EM, SPLIT>(B, rowptr, counts, F, Gr, r0, r1, status);
}

template <int MODE, bool K1, int WARPS, int EM, bool SPLIT = false>
__global__ void __launch_bounds__(WARPS * 32, 32 / WARPS)
k_rows_const(const __grid_constant__ DevBasis B, const int64_t *rowptr, int64_t *counts, const __grid_constant__ FillArgs F, GradArgs Gr,
             int64_t r0, int64_t r1, int *status)
{
    walk_rows<MODE, K1, WARPS, EM, SPLIT>(B, rowptr, counts, F, Gr, r0, r1, status);
}

// The working copy of the tables (FillWork): warps over the rows of the pn
// squares, then over the sub-dets of both species.  Bound by its scattered
// reads of the tables (L2); it replaces two to seven of them, and the pair
// lookups, per element of that kind in every row.
template <int KV>
__global__ void __launch_bounds__(256) k_fill_prep(DevBasis B, FillArgs F, FillWork W, int *status)
{
    const int lane = threadIdx.x & 31;
    const int64_t warp = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    const int64_t n0 = B.n_sqrow, n1 = n0 + B.sp[0].n_sd, n2 = n1 + B.sp[1].n_sd;
    auto entry = [&](int64_t idx, bool neg) {                  // the sets' values (a set past the last repeats it)
        Vals<KV> r;
#pragma unroll
        for (int u = 0; u < KV; ++u) {
            const float v = __ldg(F.tbme + (int64_t)(W.k0 + min(u, W.ks - 1)) * F.tb_sk + idx * F.tb_si);
            r.v[u] = neg ? -v : v;
        }
        return r;
    };
    for (int64_t t = warp; t < n2; t += nw) {
        if (t < n0) {
            const int r = B.sqrow[t], k = r >> 16, u = r & 0xFFFF;
            const int2 g = B.pn_k[k];
            const int n = g.y;
            Vals<KV> *out = reinterpret_cast<Vals<KV> *>(W.sq) + B.pn_kq[k].x + (int64_t)u * n;
            for (int v = lane; v < n; v += 32) {
                const int lo = min(u, v), hi = max(u, v);
                out[v] = entry(g.x + lo * n - ((lo * (lo - 1)) >> 1) + (hi - lo), false);
            }
            continue;
        }
        const int s = t < n1 ? 0 : 1;
        const DevSpecies S = s ? B.sp[1] : B.sp[0];
        Vals<KV> *hi = reinterpret_cast<Vals<KV> *>(s ? W.hi[1] : W.hi[0]), *lo = reinterpret_cast<Vals<KV> *>(s ? W.lo[1] : W.lo[0]);
        float2 *dg = s ? W.d[1] : W.d[0];
        const int64_t x = t - (s ? n1 : n0), f0 = S.fw_off[x];
        const int Z = s ? B.nZ[1] : B.nZ[0], len = (int)(S.fw_off[x + 1] - f0), two = S.fw_lev[x * S.NL + S.NL - 1];
        const uint8_t *occ = (s ? B.occ[1] : B.occ[0]) + x * Z;
        for (int u = 0; u < W.ks; ++u) {
            const DF d = diag_own(B, nullptr, F, W.k0 + u, Z, [&](int i) { return S.orb_base + (int)occ[i]; }, status);
            if (lane == 0) dg[x * KV + u] = make_float2(d.hi, d.lo);
        }
        for (int i = lane; i < two; i += 32) {
            const int tb = S.fw_tb[f0 + i];
            hi[f0 + i] = entry(tb >> 1, tb & 1);
        }
        for (int i = two + lane; i < len; i += 32) {
            const int code = ~S.fw_tb[f0 + i];
            const int a = S.orb_base + (code & 0xFF), c = S.orb_base + ((code >> 8) & 0xFF);
            const DF one = onebody_term(B, F, a, c, status);
            DF own[KV];
#pragma unroll
            for (int u = 0; u < KV; ++u) own[u] = one;
            for (int j = 0; j < Z; ++j) {
                const int k = S.orb_base + (int)occ[j];
                if (k == a) continue;
                int64_t idx;
                int sg;
                if (tbme_at(B, nullptr, a, k, c, k, idx, sg)) {
                    const Vals<KV> v = entry(idx, sg < 0);
#pragma unroll
                    for (int u = 0; u < KV; ++u) own[u] = df_add(own[u], df_of(v.v[u]));
                } else if (atomicOr(status, 1) == 0) {
                    status[2] = a | (c << 16);
                    status[3] = 2 | (k << 8);
                }
            }
            Vals<KV> h, l;
#pragma unroll
            for (int u = 0; u < KV; ++u) { h.v[u] = own[u].hi; l.v[u] = own[u].lo; }
            hi[f0 + i] = h;
            lo[f0 + i] = l;
        }
    }
}

// shared memory of k_fill1: pn groups, then per warp, then the pn index table
namespace f1 {
constexpr int kg = 0;                                      // int2[64]: pn_kq
constexpr int warp0 = 64 * 8;
constexpr int w_seg = 0;                                   // int4[32], int2[32], int4[kLevels] as k_rows
constexpr int w_ext = w_seg + 32 * 16;
constexpr int w_lev = w_ext + 32 * 8;
constexpr int w_op = w_lev + kLevels * 16;                 // int32[32]: codes of the occupied protons
constexpr int w_on = w_op + 32 * 4;                        // int32[32]: and neutrons
constexpr int w_size = w_on + 32 * 4;
template <int WARPS>
constexpr int S = warp0 + WARPS * w_size;
}  // namespace f1

// read-only load of an entry, all its bytes at once
template <class T>
__device__ __forceinline__ T ld(const T *p)
{
    T r;
    if constexpr (sizeof(T) == 4) {
        const int x = __ldg(reinterpret_cast<const int *>(p));
        memcpy(&r, &x, 4);
    } else if constexpr (sizeof(T) == 8) {
        const int2 x = __ldg(reinterpret_cast<const int2 *>(p));
        memcpy(&r, &x, 8);
    } else {
        static_assert(sizeof(T) == 16, "4, 8 or 16 bytes");
        const int4 x = __ldg(reinterpret_cast<const int4 *>(p));
        memcpy(&r, &x, 16);
    }
    return r;
}

// entry at a 32-bit byte offset from a kernel argument (arrays below 4 GiB:
// one address register instead of two, no 64-bit address arithmetic)
template <class T>
__device__ __forceinline__ T at_byte(const void *base, unsigned off)
{
    return ld(reinterpret_cast<const T *>(reinterpret_cast<const char *>(base) + off));
}

constexpr int kW = 2;             // pn windows of 32 elements in flight in k_fill1

// The fill of up to KV sets from their working copy: the walk of k_rows, every element
// one read of a value (two-moves: contiguous; pn: one gather from the squares),
// one-moves and the diagonal the prepared own-species sum plus the terms over
// the other species.  Reading the table itself in every row (pair lookups, a
// gather per spectator) took 364 us at 4+4 Nmax=4 and 8.5 ms at 4+4 Nmax=6;
// this form 298 us and 7.1 ms with its preparation, and, with rows of 16 proton
// sub-dets side by side and rows taken by next_row, 281 us and 5.6 ms.  At 3+3
// Nmax=6 it issues 6.1 warp instructions per stored nonzero (70 % of the issue slots;
// 10.9 before the groups); the pn loop is 60 % of the time, waiting on L2 for the
// members, moves and values of its windows.
template <int WARPS, int KV>
__global__ void __launch_bounds__(WARPS * 32, 32 / WARPS)
k_fill1(DevBasis B, const int64_t *rowptr, FillArgs F, FillWork W, int64_t r0, int64_t r1, int *status)
{
    constexpr int kThreads = WARPS * 32;
    extern __shared__ __align__(16) unsigned char sb[];
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const unsigned lt = (1u << lane) - 1;
    const DevSpecies &SP = B.sp[0], &SN = B.sp[1];
    const int T = B.pn_T, Zp = B.nZ[0], Zn = B.nZ[1];
    int2 *KQ = sptr<int2>(sb, f1::kg);
    int16_t *S = sptr<int16_t>(sb, f1::S<WARPS>);
    __shared__ int taken;
    if (tid == 0) taken = WARPS;
    for (int i = tid; i < SP.n_orb * T; i += kThreads) S[i] = B.pn_s[i];
    for (int i = tid; i < 64; i += kThreads) KQ[i] = B.pn_kq[i];
    __syncthreads();
    const int64_t sbase = F.sharded ? rowptr[F.shard_row] : 0;
    const int64_t nnz = F.sharded ? rowptr[r1] - sbase : rowptr[B.dim];
    unsigned char *wb = sb + f1::warp0 + wid * f1::w_size;
    int4 *w_seg = sptr<int4>(wb, f1::w_seg), *w_lev = sptr<int4>(wb, f1::w_lev);
    int2 *w_ext = sptr<int2>(wb, f1::w_ext);
    int *w_op = sptr<int>(wb, f1::w_op), *w_on = sptr<int>(wb, f1::w_on);
    constexpr int NW = KV == 1 ? kW : 1;                        // windows in flight
    const int64_t es = F.em ? F.K : 1, kst = F.em ? 1 : nnz;    // value of set k at row position e: val[e * es + k * kst]
    const Vals<KV> *sq = reinterpret_cast<const Vals<KV> *>(W.sq);
    const bool cols = W.k0 == 0;                                // (a later pass of the same fill leaves the columns)
    auto put = [&](int32_t *col, float *val, int e, int c, const Vals<KV> &v, bool neg) {
        if (cols) __stcs(col + e, c);
        const int sm = neg ? (int)0x80000000 : 0;
        if (KV == 4 && F.vec4 && F.em) {                        // four sets, element-major: one store
            const float4 r = make_float4(__int_as_float(__float_as_int(v.v[0]) ^ sm), __int_as_float(__float_as_int(v.v[KV > 1 ? 1 : 0]) ^ sm),
                                         __int_as_float(__float_as_int(v.v[KV > 2 ? 2 : 0]) ^ sm),
                                         __int_as_float(__float_as_int(v.v[KV > 2 ? 3 : 0]) ^ sm));
            __stcs(reinterpret_cast<float4 *>(val + (int64_t)e * es), r);
            return;
        }
#pragma unroll
        for (int u = 0; u < KV; ++u)
            if (KV == 1 || u < W.ks) __stcs(val + e * es + u * kst, __int_as_float(__float_as_int(v.v[u]) ^ sm));
    };
    const int P = term_lanes(Zp, Zn), sub = lane / P, li = lane % P, per = 32 / P;

    const bool walk = B.walk && r0 == 0 && r1 == B.dim;         // (a range of rows is taken in row order)
    for (int64_t place = first_row<WARPS>(r0, wid); place < r1; place = next_row<WARPS>(place, r0, r1, &taken, lane)) {
        const int2 at_row = walk ? B.walk[place] : make_int2(B.row_p[place], (int)place);
        const int p = at_row.x;
        const int64_t row = at_row.y;
        const ProtonRec PR = B.prec[p];
        const int n = (int)(row - PR.colb);
        const NeutronRec NR = B.nrec[n];
        const int64_t e0 = rowptr[row] - sbase;
        const int rowlen = (int)(min(rowptr[row + 1] - sbase, nnz) - e0);
        int32_t *col = F.col + e0;
        float *val = F.val + e0 * es + W.k0 * kst;
        const int16_t *dirn = B.dir + (int64_t)n * B.dir_len;
        const int cA1 = max(0, dirn[PR.dirA] - NR.self), cA2 = SN.fw_lev[(int64_t)n * SN.NL + PR.levA];
        int pos = 1 + cA1 + cA2;
        if (pos > rowlen) {
            if (lane == 0) atomicOr(status, 2);
            continue;
        }
        if (lane < Zp) w_op[lane] = B.occ_code[0][(int64_t)p * Zp + lane];
        if (lane < Zn) w_on[lane] = B.occ_code[1][(int64_t)n * Zn + lane];
        const int2 *recn = SN.fw_rec + NR.fw, *recp = SP.fw_rec + PR.fw;
        const Vals<KV> *vn = reinterpret_cast<const Vals<KV> *>(W.hi[1]) + NR.fw, *vp = reinterpret_cast<const Vals<KV> *>(W.hi[0]) + PR.fw;
        const int2 *n1row = B.n1p + NR.n1, *l1row = B.l1 + PR.l1;
        const unsigned l1o = (unsigned)PR.l1 * 8u, n1o = (unsigned)NR.n1 * 8u, fpo = (unsigned)(PR.fw + PR.fwlen) * 8u;
        __syncwarp();

        // diagonal
        {
            DF acc[KV];
#pragma unroll
            for (int u = 0; u < KV; ++u) acc[u] = df_of(0.f);
            for (int i = sub; i < Zp; i += per)
                if (li < Zn) {
                    const Vals<KV> v = ld(sq + pn_square_at(KQ, S, T, w_op[i], w_on[li]));
#pragma unroll
                    for (int u = 0; u < KV; ++u) acc[u] = df_add(acc[u], df_of(v.v[u]));
                }
            Vals<KV> r;
#pragma unroll
            for (int u = 0; u < KV; ++u) {
                acc[u] = warp_sum(acc[u], 32);
                const float2 dp = W.d[0][(int64_t)p * KV + u], dn = W.d[1][(int64_t)n * KV + u];
                r.v[u] = df_round(df_add(acc[u], df_add(DF{dp.x, dp.y}, DF{dn.x, dn.y})));
            }
            if (lane == 0) put(col, val, 0, (int32_t)row, r, false);
        }
        // A: neutron two-moves
        for (int t = lane; t < cA2; t += 32) {
            const int2 rc = ld(recn + t);
            put(col, val, 1 + t + (rc.y & 0xFFFFFF), PR.colb + rc.x, ld(vn + t), false);
        }
        // B: p's groups, a lane each
        int c1 = 0;                                             // proton one-moves with n kept
        for (int g0 = 0; g0 < PR.ng; g0 += 32) {
            int4 gr = make_int4(0, 0, 0, 0);
            if (g0 + lane < PR.ng) gr = B.grp[PR.g0 + g0 + lane];
            const int n1c = (unsigned)gr.x >> 16, s0 = dirn[gr.y & 0xFFFF], len = dirn[(unsigned)gr.y >> 16] - s0;
            const int self = (gr.w & 0xFF) > NR.N ? 1 : 0;                  // own class and N_n <= L_q
            const int npn = n1c * len, tot = npn + self * (n1c + gr.z);
            int itot = tot, ipn = npn;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const int o1 = __shfl_up_sync(0xffffffffu, itot, d), o2 = __shfl_up_sync(0xffffffffu, ipn, d);
                if (lane >= d) { itot += o1; ipn += o2; }
            }
            const int Tall = __shfl_sync(0xffffffffu, itot, 31), Tpn = __shfl_sync(0xffffffffu, ipn, 31);
            if (pos + Tall > rowlen) {
                if (lane == 0) atomicOr(status, 2);
                break;
            }
            const int at0 = pos + itot - tot, st = ipn - npn, m1 = gr.x & 0xFFFF;
            const int ins = NR.self - s0;                                   // where n sorts in the segment
            const int c = at0 - m1 * (len + 1) - (gr.w >> 8);
            const unsigned ne = __ballot_sync(0xffffffffu, npn > 0);
            if (npn > 0) {
                const int j = __popc(ne & lt);
                w_seg[j] = make_int4(st, (int)(0xFFFFFFFFu / (unsigned)len), m1, self ? c : at0 - st);
                w_ext[j] = make_int2(s0 | len << 16, self ? ins : -1);
            }
            int c2 = 0;
            if (g0 == 0) {                                      // own-class groups come first, at most kLevels
                if (gr.w) w_lev[((B.Nlim - (gr.w & 0xFF) + 1) - SP.N0) >> 1] = make_int4(c, len + 1, ins, 0);
                c1 = __reduce_add_sync(0xffffffffu, self * n1c);
                c2 = __reduce_add_sync(0xffffffffu, self * gr.z);
            }
            __syncwarp();
            for (int t = lane; t < c2; t += 32) {               // pp two-moves: a prefix of p's list
                const int2 rc = ld(recp + t);
                const int4 lv = w_lev[rc.y >> 24];
                put(col, val, lv.x + t + (rc.y & 0xFFFFFF) * lv.y, rc.x + n, ld(vp + t), false);
            }
            // pn elements of all groups, flattened as in k_rows, kW windows of 32
            // at a time so that their chains of loads (member and neutron move, then
            // the value) overlap; lanes past the end repeat the last element's loads
            const unsigned le = (2u << lane) - 1u;                 // bits 0..lane
            int before = -1;                                       // pn groups started before the window, less one
            for (int w0 = 0; w0 < Tpn; w0 += 32 * NW) {
                int2 q[NW], ent[NW];
                int at[NW];
#pragma unroll
                for (int u = 0; u < NW; ++u) {
                    const int w = w0 + 32 * u;
                    const unsigned mk = __reduce_or_sync(0xffffffffu, npn > 0 && (unsigned)(st - w) < 32u ? 1u << (st - w) : 0u);
                    const int j = before + __popc(mk & le), e = min(w + lane, Tpn - 1);
                    before += __popc(mk);
                    const int4 sg4 = w_seg[j];
                    const int2 sx = w_ext[j];
                    const int rel = e - sg4.x, ln = (unsigned)sx.x >> 16;
                    int qi = (int)__umulhi((unsigned)rel, (unsigned)sg4.y), k = rel - qi * ln;   // at most one short
                    if (k >= ln) { ++qi; k -= ln; }
                    const unsigned i1 = sg4.z + qi;
                    q[u] = at_byte<int2>(B.l1, l1o + i1 * 8);
                    ent[u] = at_byte<int2>(B.n1p, n1o + ((sx.x & 0xFFFF) + k) * 8);
                    at[u] = sg4.w + e;
                    if (sx.y >= 0)                                 // n itself is among the partners
                        at[u] = sg4.w + i1 * (ln + 1) + (at_byte<int2>(SP.fw_rec, fpo - 8 - i1 * 8).y & 0xFFFFFF) + k +
                                (k >= sx.y ? 1 : 0);
                }
                Vals<KV> v[NW];
#pragma unroll
                for (int u = 0; u < NW; ++u)
                    v[u] = at_byte<Vals<KV>>(W.sq, (unsigned)pn_square_at(KQ, S, T, q[u].y, ent[u].y) * (4u * KV));
#pragma unroll
                for (int u = 0; u < NW; ++u) {
                    if (w0 + 32 * u + lane >= Tpn) continue;
                    put(col, val, at[u], q[u].x + ent[u].x, v[u], ((q[u].y >> 16) ^ (ent[u].y >> 26)) & 1);
                }
            }
            __syncwarp();
            pos += Tall;
        }
        // one-moves of either species: P lanes an element, one per particle of
        // the other species
        for (int t0 = 0; t0 < cA1 + c1; t0 += per) {
            const int t = t0 + sub;
            const bool act = t < cA1 + c1, neu = t < cA1;
            int lc = 0, nc = 0, e = 0, j = 0, sgn = 0;
            int64_t slot = 0;
            if (act && neu) {
                const int2 ent = n1row[NR.self + t];
                slot = NR.fwlen - 1 - t;
                e = 1 + t + (recn[slot].y & 0xFFFFFF);
                j = PR.colb + ent.x;
                sgn = (ent.y >> 26) & 1;
                nc = ent.y;
                if (li < Zp) lc = w_op[li];
            } else if (act) {
                const int i1 = t - cA1;
                const int2 q = l1row[i1];
                slot = PR.fwlen - 1 - i1;
                const int o = recp[slot].y;
                const int4 lv = w_lev[o >> 24];
                e = lv.x + i1 * lv.y + (o & 0xFFFFFF) + lv.z;
                j = q.x + n;
                sgn = (q.y >> 16) & 1;
                lc = q.y;
                if (li < Zn) nc = w_on[li];
            }
            const bool has = act && li < (neu ? Zp : Zn);
            Vals<KV> v{};
            if (has) v = ld(sq + pn_square_at(KQ, S, T, lc, nc));
            DF sum[KV];
#pragma unroll
            for (int u = 0; u < KV; ++u) sum[u] = warp_sum(df_of(v.v[u]), P);
            if (act && li == 0) {
                slot += neu ? NR.fw : PR.fw;
                const Vals<KV> h = ld(reinterpret_cast<const Vals<KV> *>(neu ? W.hi[1] : W.hi[0]) + slot),
                               l = ld(reinterpret_cast<const Vals<KV> *>(neu ? W.lo[1] : W.lo[0]) + slot);
                Vals<KV> r;
#pragma unroll
                for (int u = 0; u < KV; ++u) r.v[u] = df_round(df_add(sum[u], DF{h.v[u], l.v[u]}));
                put(col, val, e, j, r, sgn);
            }
        }
        __syncwarp();
    }
}

// ---- adjoint of one vector
//
// Every sum here is of integers, so its parts may be added in any grouping:
//   own species   an element that moves one species only (two-moves; the
//                 own-species spectators of one-moves; the own part of the
//                 diagonal) uses the same table entry whatever the other species
//                 does.  k_grad_pairs sums psi psi over the common partners of
//                 each forward pair (two contiguous runs of psi) and adds once
//                 per pair instead of once per row: a tenth of all adds;
//   the rest      (pn moves, and the other species' terms of one-moves and of
//                 the diagonal) k_grad1 adds per row.
// For the neutrons the vector is copied neutron-major, so that their runs are
// contiguous too.  k_grad1 adds into the pn groups as full squares (folded at the
// end): the entries of a proton move and one neutron orbital are contiguous there,
// and the limit is the number of 32-byte sectors of the atomic adds (4+4 Nmax=6:
// 8.1 ms in the row kernel, 7.7 into the packed triangles, 6.2 into the squares).

// The partners of the sub-dets of species s: other-species sub-dets beg[x] ..
// beg[x] + lev[x * NL + l] - 1 pair with every same-class sub-det of level l (a
// prefix of the class, ascending in N); cnt[x] is x's own count.
struct Partners {
    const int32_t *beg[2], *lev[2];
    const int64_t *base[2];                // first place of x's run in the vector of its species' order
    const long long *psi[2];               // the vector proton-major (as given) and neutron-major
};

__global__ void k_partners(DevBasis B, SpeciesBuild S0, SpeciesBuild S1, int s, int twoM, int32_t *beg, int32_t *lev, int64_t *cnt)
{
    const DevSpecies &X = B.sp[s];
    const SpeciesBuild &Sx = s ? S1 : S0, &So = s ? S0 : S1;
    for (int x = blockIdx.x * blockDim.x + threadIdx.x; x < X.n_sd; x += gridDim.x * blockDim.x) {
        const int M = twoM - Sx.M2[x], par = (B.Nlim - Sx.N[x]) & 1;
        auto below = [&](int par_, int N) {                  // sub-dets ordered (2M, parity, N) before (M, par_, N)
            int lo = 0, hi = So.n_sd;
            while (lo < hi) {
                const int mid = (lo + hi) >> 1, m = So.M2[mid], q = So.N[mid], r = q & 1;
                if (m != M ? m < M : r != par_ ? r < par_ : q < N) lo = mid + 1; else hi = mid;
            }
            return lo;
        };
        const int b0 = below(par, -1), px = (Sx.N[x] - X.N0) & 1;
        beg[x] = b0;
        for (int l = 0; l < X.NL; ++l) {
            const int c = below(par, B.Nlim - (X.N0 + 2 * l + px) + 1) - b0;
            lev[x * X.NL + l] = c > 0 ? c : 0;
            if (l == (Sx.N[x] - X.N0) >> 1) cnt[x] = c;
        }
    }
}

// out[base[n] + p - beg[n]] = psi[row of (p, n)]
__global__ void k_psi_neutron_major(DevBasis B, const int32_t *beg, const int64_t *base, const long long *psi, long long *out)
{
    for (int64_t row = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; row < B.dim; row += (int64_t)gridDim.x * blockDim.x) {
        const int p = B.row_p[row], n = (int)(row - B.prec[p].colb);
        out[base[n] + p - beg[n]] = psi[row];
    }
}

// One block per sub-det x (the lowest ones have thousands of pairs with hundreds
// of partners), eight lanes per forward pair (x, y): the sum over their common
// partners of psi psi, added to the pair's table entry (two-move) or to its
// own-species spectator entries (one-move).
__global__ void __launch_bounds__(256) k_grad_pairs(DevBasis B, Partners Pt, unsigned long long *acc, int *status)
{
    const int tid = threadIdx.x, lane = tid & 31, li = tid & 7;
    const int64_t n0 = B.sp[0].n_sd, n1 = n0 + B.sp[1].n_sd;
    for (int64_t t = blockIdx.x; t < n1; t += gridDim.x) {
        const int s = t < n0 ? 0 : 1;
        const DevSpecies S = s ? B.sp[1] : B.sp[0];
        const int64_t x = t - (s ? n0 : 0), f0 = S.fw_off[x];
        const int Z = s ? B.nZ[1] : B.nZ[0], len = (int)(S.fw_off[x + 1] - f0), two = S.fw_lev[x * S.NL + S.NL - 1];
        const uint8_t *occ = (s ? B.occ[1] : B.occ[0]) + x * Z;
        const int32_t *lev = (s ? Pt.lev[1] : Pt.lev[0]) + x * S.NL;
        const int64_t *base = s ? Pt.base[1] : Pt.base[0];
        const long long *psi = s ? Pt.psi[1] : Pt.psi[0], *px = psi + base[x];
        const int nb = s ? 0 : B.nb[x];
        if (tid < 32) {                                         // own part of the diagonal: weight 1, every partner of x
            const int c = (int)(base[x + 1] - base[x]);
            long long sum = 0;
            for (int i = lane; i < c; i += 32) sum += __mul64hi(px[i], px[i]) >> 2;
            for (int d = 16; d > 0; d >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, d);
            for (int l = lane; l < Z * (Z - 1) / 2; l += 32) {
                int i, j, sg;
                int64_t idx;
                pair_of(l, Z, i, j);
                const int a = S.orb_base + occ[i], b = S.orb_base + occ[j];
                if (tbme_at(B, nullptr, a, b, a, b, idx, sg)) atomicAdd(acc + idx, (unsigned long long)(sg < 0 ? -sum : sum));
                else if (atomicOr(status, 1) == 0) { status[2] = a | (b << 16); status[3] = 1; }
            }
        }
        for (int e0 = 0; e0 < len; e0 += 32) {
            const int e = e0 + (tid >> 3);
            const bool on = e < len;
            long long sum = 0;
            int tb = 0;
            if (on) {
                const int2 rc = S.fw_rec[f0 + e];
                tb = S.fw_tb[f0 + e];
                const long long *py = psi + (s ? base[rc.x] : (int64_t)(rc.x + nb));
                const int c = lev[rc.y >> 24];
                for (int i = li; i < c; i += 8) sum += __mul64hi(px[i], py[i]) >> 1;
            }
            for (int d = 4; d > 0; d >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, d);
            if (!on) continue;
            if (e < two) {
                if (li == 0) atomicAdd(acc + (tb >> 1), (unsigned long long)(tb & 1 ? -sum : sum));
                continue;
            }
            const int code = ~tb, a = S.orb_base + (code & 0xFF), c = S.orb_base + ((code >> 8) & 0xFF);
            for (int i = li; i < Z; i += 8) {
                const int k = S.orb_base + occ[i];
                if (k == a) continue;
                int64_t idx;
                int sg;
                if (tbme_at(B, nullptr, a, k, c, k, idx, sg))
                    atomicAdd(acc + idx, (unsigned long long)(((code >> 16) & 1) != (sg < 0) ? -sum : sum));
                else if (atomicOr(status, 1) == 0) {
                    status[2] = a | (c << 16);
                    status[3] = 2 | (k << 8);
                }
            }
        }
    }
}

// acc of the table entries of the pn groups += the squares' entries: (u, v) and
// (v, u) are one; one warp per row of a square
__global__ void __launch_bounds__(256) k_grad_fold(DevBasis B, const unsigned long long *sq, unsigned long long *acc)
{
    const int lane = threadIdx.x & 31;
    const int64_t warp = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5, nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t t = warp; t < B.n_sqrow; t += nw) {
        const int r = B.sqrow[t], k = r >> 16, u = r & 0xFFFF;
        const int2 g = B.pn_k[k];
        const int n = g.y;
        const unsigned long long *s = sq + B.pn_kq[k].x;
        unsigned long long *o = acc + g.x + (int64_t)u * n - ((int64_t)u * (u - 1)) / 2 - u;
        for (int v = u + lane; v < n; v += 32) {
            unsigned long long x = s[(int64_t)u * n + v];
            if (v > u) x += s[(int64_t)v * n + u];
            o[v] += x;
        }
    }
}

// The walk of k_fill1 without places: every (member, neutron move) pair of the
// row's groups, and the other species' terms of its one-moves and diagonal.
template <int WARPS>
__global__ void __launch_bounds__(WARPS * 32, 32 / WARPS)
k_grad1(DevBasis B, const long long *psi, unsigned long long *acc)
{
    constexpr int kThreads = WARPS * 32;
    extern __shared__ __align__(16) unsigned char sb[];
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const unsigned lt = (1u << lane) - 1, le = (2u << lane) - 1u;
    const DevSpecies &SP = B.sp[0];
    const int T = B.pn_T, Zp = B.nZ[0], Zn = B.nZ[1];
    int2 *KG = sptr<int2>(sb, f1::kg);
    int16_t *S = sptr<int16_t>(sb, f1::S<WARPS>);
    __shared__ int taken;
    if (tid == 0) taken = WARPS;
    for (int i = tid; i < SP.n_orb * T; i += kThreads) S[i] = B.pn_s[i];
    for (int i = tid; i < 64; i += kThreads) KG[i] = B.pn_kq[i];
    __syncthreads();
    unsigned char *wb = sb + f1::warp0 + wid * f1::w_size;
    int4 *w_seg = sptr<int4>(wb, f1::w_seg);
    int *w_s0 = sptr<int>(wb, f1::w_ext);
    int *w_op = sptr<int>(wb, f1::w_op), *w_on = sptr<int>(wb, f1::w_on);
    const int P = term_lanes(Zp, Zn), sub = lane / P, li = lane % P, per = 32 / P;
    auto add = [&](int l1, int n1, long long q) {
        const int idx = pn_square_at(KG, S, T, l1, n1);
        atomicAdd(acc + idx, (unsigned long long)(((l1 >> 16) ^ (n1 >> 26)) & 1 ? -q : q));
    };
    for (int64_t place = first_row<WARPS>(0, wid); place < B.dim; place = next_row<WARPS>(place, 0, B.dim, &taken, lane)) {
        const int2 at_row = B.walk ? B.walk[place] : make_int2(B.row_p[place], (int)place);
        const int p = at_row.x;
        const int64_t row = at_row.y;
        const ProtonRec PR = B.prec[p];
        const int n = (int)(row - PR.colb);
        const NeutronRec NR = B.nrec[n];
        const long long pr = psi[row];
        const int16_t *dirn = B.dir + (int64_t)n * B.dir_len;
        const int cA1 = max(0, dirn[PR.dirA] - NR.self);
        if (lane < Zp) w_op[lane] = B.occ_code[0][(int64_t)p * Zp + lane];
        if (lane < Zn) w_on[lane] = B.occ_code[1][(int64_t)n * Zn + lane];
        const unsigned l1o = (unsigned)PR.l1 * 8u, n1o = (unsigned)NR.n1 * 8u;
        __syncwarp();
        {                                                       // diagonal, w = 1
            const long long q = __mul64hi(pr, pr) >> 2;
            for (int i = sub; i < Zp; i += per)
                if (li < Zn) add(w_op[i], w_on[li], q);
        }
        int c1 = 0;                                             // proton one-moves with n kept
        for (int g0 = 0; g0 < PR.ng; g0 += 32) {
            int4 gr = make_int4(0, 0, 0, 0);
            if (g0 + lane < PR.ng) gr = B.grp[PR.g0 + g0 + lane];
            const int n1c = (unsigned)gr.x >> 16, s0 = dirn[gr.y & 0xFFFF], len = dirn[(unsigned)gr.y >> 16] - s0;
            if (g0 == 0) c1 = __reduce_add_sync(0xffffffffu, (gr.w & 0xFF) > NR.N ? n1c : 0);
            const int npn = n1c * len;
            int ipn = npn;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const int o = __shfl_up_sync(0xffffffffu, ipn, d);
                if (lane >= d) ipn += o;
            }
            const int Tpn = __shfl_sync(0xffffffffu, ipn, 31), st = ipn - npn;
            const unsigned ne = __ballot_sync(0xffffffffu, npn > 0);
            if (npn > 0) {
                const int j = __popc(ne & lt);
                w_seg[j] = make_int4(st, (int)(0xFFFFFFFFu / (unsigned)len), gr.x & 0xFFFF, len);
                w_s0[j] = s0;
            }
            __syncwarp();
            int before = -1;
            for (int w0 = 0; w0 < Tpn; w0 += 32 * kW) {         // as in k_fill1
                int2 q[kW], ent[kW];
                long long v[kW];
#pragma unroll
                for (int u = 0; u < kW; ++u) {
                    const int w = w0 + 32 * u;
                    const unsigned mk = __reduce_or_sync(0xffffffffu, npn > 0 && (unsigned)(st - w) < 32u ? 1u << (st - w) : 0u);
                    const int j = before + __popc(mk & le), e = min(w + lane, Tpn - 1);
                    before += __popc(mk);
                    const int4 sg4 = w_seg[j];
                    const int rel = e - sg4.x;
                    int qi = (int)__umulhi((unsigned)rel, (unsigned)sg4.y), k = rel - qi * sg4.w;   // at most one short
                    if (k >= sg4.w) { ++qi; k -= sg4.w; }
                    q[u] = at_byte<int2>(B.l1, l1o + (unsigned)(sg4.z + qi) * 8u);
                    ent[u] = at_byte<int2>(B.n1p, n1o + (unsigned)(w_s0[j] + k) * 8u);
                }
#pragma unroll
                for (int u = 0; u < kW; ++u) v[u] = __ldg(psi + (q[u].x + ent[u].x));
#pragma unroll
                for (int u = 0; u < kW; ++u)
                    if (w0 + 32 * u + lane < Tpn) add(q[u].y, ent[u].y, __mul64hi(pr, v[u]) >> 1);
            }
            __syncwarp();
        }
        for (int t0 = 0; t0 < cA1 + c1; t0 += per) {            // one-moves: P lanes an element
            const int t = t0 + sub;
            if (t >= cA1 + c1) continue;
            const bool neu = t < cA1;
            const int2 m = neu ? B.n1p[NR.n1 + NR.self + t] : B.l1[PR.l1 + t - cA1];
            if (li >= (neu ? Zp : Zn)) continue;
            const long long q = __mul64hi(pr, psi[neu ? PR.colb + m.x : m.x + n]) >> 1;
            add(neu ? w_op[li] : m.y, neu ? m.y : w_on[li], q);
        }
        __syncwarp();
    }
}

// Count pass: for row (p, n), 1 for the diagonal + n's forward same-class
// neighbours inside p's range + the sum over p's groups of members x segment
// length (+ members and two-moves where n itself is a partner).  Equal to the
// walk's count.  Each row is a chain of dependent loads (row -> p -> n ->
// directory), so a warp takes 32 / G rows at a time, G lanes each, to keep
// that many chains in flight; every warp-wide intrinsic is reached by all 32
// lanes.
template <int G>
__global__ void __launch_bounds__(256) k_count(DevBasis B, int64_t *counts, int64_t r0, int64_t r1)
{
    constexpr int R = 32 / G;
    const int lane = threadIdx.x & 31, g = lane / G, li = lane % G;
    const unsigned full = 0xffffffffu;
    const int64_t gw = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    const DevSpecies &SN = B.sp[1];
    for (int64_t base = r0 + gw * R; base < r1; base += nw * R) {      // uniform over the warp
        const int64_t row = base + g;
        const bool live = row < r1;
        int acc = 0;
        if (live) {
            const int p = B.row_p[row];
            const ProtonRec PR = B.prec[p];
            const int n = (int)(row - PR.colb);
            const int16_t *dirn = B.dir + (int64_t)n * B.dir_len;
            const int Nn = SN.N[n];
            if (li == 0)
                acc = 1 + max(0, dirn[PR.dirA] - SN.n1_self[n]) + SN.fw_lev[(int64_t)n * SN.NL + PR.levA];
#pragma unroll 4
            for (int q = li; q < PR.ng; q += G) {
                const int4 gr = B.grp[PR.g0 + q];
                const int n1c = (unsigned)gr.x >> 16;
                acc += n1c * (dirn[(unsigned)gr.y >> 16] - dirn[gr.y & 0xFFFF]);
                if ((gr.w & 0xFF) > Nn) acc += n1c + gr.z;
            }
        }
#pragma unroll
        for (int o = G / 2; o > 0; o >>= 1) acc += __shfl_xor_sync(full, acc, o);
        if (live && li == 0) counts[row] = acc;
    }
}

// Raise a kernel's dynamic shared-memory limit on a device once per size, so
// that later calls (inside a stream capture, say) only launch.
cudaError_t raise_smem_limit(const void *kern, int dev, int bytes)
{
    static std::mutex mu;
    static std::map<std::pair<const void *, int>, int> raised;
    std::lock_guard<std::mutex> lock(mu);
    int &have = raised[{kern, dev}];
    if (bytes <= have) return cudaSuccess;
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e == cudaSuccess) have = bytes;
    return e;
}

// Parts that the elements of a row are filled in, a CTA each: the diagonal and the
// neutron moves; the proton moves; the pn elements (the last two together where two
// parts are all that the GPU holds at once).  The chain of one warp that fills a row
// takes most of the time of a fill of few rows, whose CTAs leave SMs idle.  us, one
// part / three: 800 rows of 3+3 Nmax=2 16.4 / 12.3 with one set, 20.5 / 14.3 with four.
inline int row_parts(int64_t ctas, int64_t held) { return 3 * ctas <= held ? 3 : 2 * ctas <= held ? 2 : 1; }

template <int MODE, int WARPS>
int launch_rows_w(const cih_basis &b, const int64_t *rowptr, int64_t *counts, const FillArgs &F, const GradArgs &G,
                  cudaStream_t st, bool dry, int64_t r0, int64_t r1)
{
    const DevBasis &D = b.dev;
    const size_t smem = MODE == 0 ? (size_t)sm::S<WARPS> : smem_bytes<WARPS>(D.sp[0].n_orb * D.pn_T);
    int dev = 0, sms = 148;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    auto go = [&](auto kern) -> int {
        cudaError_t ee = raise_smem_limit((const void *)kern, dev, (int)smem);
        if (ee != cudaSuccess) return cuda_fail(ee, "row kernel shared memory");
        if (dry) return CIH_OK;                              // set-up only, no launch
        int per_sm = 0;
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, WARPS * 32, smem);
        per_sm = std::max(per_sm, 1);
        if (b.launch_ctas > 0) per_sm = std::min(per_sm, b.launch_ctas);
        const int64_t want = (r1 - r0 + WARPS - 1) / WARPS;
        const int grid = (int)std::max<int64_t>(1, std::min<int64_t>((int64_t)sms * per_sm, want));
        const int parts = MODE == 1 ? row_parts(want, (int64_t)sms * per_sm) : 1;
        count_launches(1);
        kern<<<dim3(grid, parts), WARPS * 32, smem, st>>>(D, rowptr, counts, F, G, r0, r1, b.dev_status);
        ee = cudaGetLastError();
        return ee == cudaSuccess ? CIH_OK : cuda_fail(ee, "row kernel launch");
    };
    const bool k1 = (MODE == 1 && F.K == 1) || (MODE == 2 && G.K == 1);   // one set / one vector
    const int L4 = F.K >> 2;
    const bool em = MODE == 1 && F.K >= kFillSets && F.em && F.vec4 && (L4 > 32 ? L4 % 32 == 0 : 32 % L4 == 0);
    if constexpr (MODE == 1) {
        // element-major K sets: warp-cooperative writes; 64 is the batched configuration's set count
        if (em) return F.K == 64 ? go(k_rows<MODE, false, WARPS, 64>) : go(k_rows<MODE, false, WARPS, 1>);
    }
    if constexpr (MODE == 1) {
        if (F.tol_one > 0.f) return k1 ? go(k_rows_const<MODE, true, WARPS, 0, true>) : go(k_rows_const<MODE, false, WARPS, 0, true>);
    }
    if constexpr (MODE == 1) {
        if (k1) return go(k_rows_const<MODE, true, WARPS, 0>);
    }
    if constexpr (MODE == 2) {
        if (k1) return go(k_rows<MODE, true, WARPS, 0>);
    }
    return go(k_rows<MODE, false, WARPS, 0>);
}

template <int MODE>
int launch_rows(const cih_basis &b, const int64_t *rowptr, int64_t *counts, const FillArgs &F, const GradArgs &G,
                cudaStream_t st, bool dry = false, int64_t r0 = 0, int64_t r1 = -1)
{
    if (r1 < 0) r1 = b.dim;
    if (b.dim == 0 || (!dry && r1 <= r0)) return CIH_OK;
    const DevBasis &D = b.dev;
    if (D.A > kMaxA || D.A - 1 > 32) return fail(CIH_ERR_UNSUPPORTED, "more than 33 particles");
    if (D.tbme_len > INT32_MAX) return fail(CIH_ERR_UNSUPPORTED, "two-body table above 2^31 entries");
    return b.launch_warps == 8 ? launch_rows_w<MODE, 8>(b, rowptr, counts, F, G, st, dry, r0, r1)
                               : launch_rows_w<MODE, 16>(b, rowptr, counts, F, G, st, dry, r0, r1);
}

// element-major copy of K set-major tables: out[t * K + k] = in[k * len + t]
__global__ void k_interleave(int K, int64_t len, const float *in, float *out)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < len * K; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t t = i / K;
        const int k = (int)(i - t * K);
        out[i] = in[(int64_t)k * len + t];
    }
}

__global__ void k_fix_to_double(int64_t n, const unsigned long long *acc, double *out)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        out[i] = (double)(long long)acc[i] / kFixScale;
}

}  // namespace

int launch_count(const cih_basis &b, int64_t *rowptr, cudaStream_t st)
{
    if (b.count_walk) return launch_rows<0>(b, nullptr, rowptr, FillArgs{}, GradArgs{}, st);
    if (b.dim == 0) return CIH_OK;
    int dev = 0, sms = 148, per_sm = 1;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    constexpr int G = 8;                                     // lanes per row
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_count<G>, 256, 0);
    const int64_t rows_per_block = 8 * (32 / G);
    const int grid = (int)std::max<int64_t>(
        1, std::min<int64_t>((int64_t)sms * std::max(per_sm, 1), (b.dim + rows_per_block - 1) / rows_per_block));
    count_launches(1);
    k_count<G><<<grid, 256, 0, st>>>(b.dev, rowptr, 0, b.dim);
    const cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? CIH_OK : cuda_fail(e, "count launch");
}

int launch_scan(const cih_basis &b, int64_t *rowptr, cudaStream_t st)
{
    return exclusive_scan_i64(rowptr, b.dim, b.scan_scratch, b.scan_scratch_len, st);
}

namespace {

// Layout of the working copy of kv sets: the squares, the slots, then the pairs of
// the diagonal, each at a multiple of 16 bytes.
size_t work_floats(const cih_basis &b, int kv)
{
    auto up = [](int64_t n) { return (n + 3) / 4 * 4; };
    return (size_t)(up(b.sq_total * kv) + 2 * up(b.fw_total[0] * kv) + 2 * up(b.fw_total[1] * kv) +
                    up(2 * b.s[0].n_sd * kv) + up(2 * b.s[1].n_sd * kv));
}

FillWork work_at(const cih_basis &b, float *p, int kv, int k0, int ks)
{
    auto take = [&](int64_t n) { float *q = p; p += (n + 3) / 4 * 4; return q; };
    FillWork w;
    w.sq = take(b.sq_total * kv);
    for (int s = 0; s < 2; ++s) {
        w.hi[s] = take(b.fw_total[s] * kv);
        w.lo[s] = take(b.fw_total[s] * kv);
    }
    for (int s = 0; s < 2; ++s) w.d[s] = reinterpret_cast<float2 *>(take(2 * b.s[s].n_sd * kv));
    w.k0 = k0;
    w.ks = ks;
    return w;
}

// k_fill1 takes 32-bit byte offsets and keeps at most 32 particles of a species
bool fill1_fits(const cih_basis &b, int kv)
{
    const int64_t most = (int64_t)1 << 32;
    for (int s = 0; s < 2; ++s)
        if (b.fw_total[s] * 8 >= most || b.n1_total[s] * 8 >= most) return false;
    return b.sq_total * 4 * kv < most && b.dev.A - 1 <= 32 && b.dev.nZ[0] <= 32 && b.dev.nZ[1] <= 32 && b.dim > 0;
}

template <int WARPS, int KV>
int launch_fill1_w(const cih_basis &b, const int64_t *rowptr, const FillArgs &F, const FillWork &W, cudaStream_t st, bool dry,
                   int64_t r0, int64_t r1)
{
    const size_t smem = (size_t)f1::S<WARPS> + ((size_t)b.dev.sp[0].n_orb * b.dev.pn_T * 2 + 15) / 16 * 16;
    int dev = 0, sms = 148;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaError_t e = raise_smem_limit((const void *)k_fill1<WARPS, KV>, dev, (int)smem);
    if (e != cudaSuccess) return cuda_fail(e, "fill shared memory");
    if (dry) return CIH_OK;
    int per_sm = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_fill1<WARPS, KV>, WARPS * 32, smem);
    per_sm = std::max(per_sm, 1);
    if (b.launch_ctas > 0) per_sm = std::min(per_sm, b.launch_ctas);
    const int64_t want = (r1 - r0 + WARPS - 1) / WARPS;
    const int grid = (int)std::max<int64_t>(1, std::min<int64_t>((int64_t)sms * per_sm, want));
    count_launches(1);
    k_fill1<WARPS, KV><<<grid, WARPS * 32, smem, st>>>(b.dev, rowptr, F, W, r0, r1, b.dev_status);
    e = cudaGetLastError();
    return e == cudaSuccess ? CIH_OK : cuda_fail(e, "fill launch");
}

int launch_fill1(const cih_basis &b, int kv, const int64_t *rowptr, const FillArgs &F, const FillWork &W, cudaStream_t st, bool dry,
                 int64_t r0, int64_t r1)
{
    if (b.launch_warps == 8)
        return kv == 1 ? launch_fill1_w<8, 1>(b, rowptr, F, W, st, dry, r0, r1)
             : kv == 2 ? launch_fill1_w<8, 2>(b, rowptr, F, W, st, dry, r0, r1) : launch_fill1_w<8, 4>(b, rowptr, F, W, st, dry, r0, r1);
    return kv == 1 ? launch_fill1_w<16, 1>(b, rowptr, F, W, st, dry, r0, r1)
         : kv == 2 ? launch_fill1_w<16, 2>(b, rowptr, F, W, st, dry, r0, r1) : launch_fill1_w<16, 4>(b, rowptr, F, W, st, dry, r0, r1);
}

int launch_prep(const cih_basis &b, int kv, const FillArgs &F, const FillWork &W, cudaStream_t st)
{
    const int64_t warps = b.dev.n_sqrow + b.s[0].n_sd + b.s[1].n_sd;
    const int grid = (int)std::max<int64_t>(1, std::min<int64_t>((warps + 7) / 8, 152 * 16));
    count_launches(1);
    if (kv == 1) k_fill_prep<1><<<grid, 256, 0, st>>>(b.dev, F, W, b.dev_status);
    else if (kv == 2) k_fill_prep<2><<<grid, 256, 0, st>>>(b.dev, F, W, b.dev_status);
    else k_fill_prep<4><<<grid, 256, 0, st>>>(b.dev, F, W, b.dev_status);
    const cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? CIH_OK : cuda_fail(e, "fill preparation");
}

// Whether a fill of K sets of `rows` of the rows goes through the working copy.  A copy
// costs its two launches and its entries once; each row gains.  Several sets
// gain more a row; from five on there are two passes, and the values of
// five to seven sets of an element, written by both, share their lines.  Measured
// against the row kernel, by rows and entries of a copy a row:
//   one set: 4,945 rows, 50 entries 0.76x; 8,500, 15 0.95x; 13,162, 85 0.93x; 17,769,
//     170 0.90x; 10,817, 34 1.12x; 14,502, 12 1.17x; 15,448, 78 0.90x; 17,040, 61 1.22x;
//     23,907, 54 1.07x; 39,421, 94 1.14x
//   two, four: 4,945, 50 0.85x, 0.91x; 6,758, 425 0.88x, 0.98x; 8,500, 15 1.12x, 1.13x;
//     10,753, 51 1.15x, 1.21x; 17,769, 170 1.06x, 1.04x
//   seven, set-major and element-major: 23,907, 54 1.11x, 0.84x; 36,498, 18 1.31x, 0.97x;
//     165,736, 82 1.36x, 0.93x; 48,917, 35 1.54x, 1.04x; 143,792, 18 1.98x, 1.15x
// A part of the rows by the same rule for its own rows, with two to four sets from
// 12,288 rows on (the copy covers all sub-dets, so few rows pay for many entries).
// Over some 500 parts (halves to fiftieths) of 20 bases, mean time over the better
// way's by this rule / always / never through the copy: one set 1.006 / 1.33 / 1.02, two
// 1.04 / 1.23 / 1.14, four 1.03 / 1.37 / 1.09, seven 1.02 / 1.81 / 1.04.
bool copy_pays(const cih_basis &b, int K, int64_t rows)
{
    const int64_t least = K == 1 ? 10240 : K > 4 ? 40960 : rows == b.dim ? 8192 : 12288;
    const int64_t entries = K == 1 ? (rows < 16384 ? 40 : 128) : K <= 4 ? 192 : 64;
    return K < kFillSets && rows >= least && fill1_fits(b, K == 1 ? 1 : K == 2 ? 2 : 4) &&
           (int64_t)work_floats(b, 1) <= entries * rows;
}
// Whether the fills of all rows of K sets go through the copy, and so the sums of
// every fill are those of its order (SPLIT)
bool fill_splits(const cih_basis &b, int K) { return copy_pays(b, K, b.dim); }

// additions a term goes through, in the row kernel's order and in k_fill1's together,
// for a one-move and for the diagonal, x 16 u^2
void split_tolerances(const cih_basis &b, FillArgs &F)
{
    auto lg = [](int x) { int l = 0; while (1 << l < x) ++l; return l; };
    auto warps = [](int x) { return (x + 31) / 32; };
    const int A = b.dev.A, Zp = b.dev.nZ[0], Z = std::max(Zp, b.dev.nZ[1]), P = std::min(lg(Z), 5);
    const int one = 1 + lg(A - 1) + std::max(Z - 1, P) + 1;
    const int pn = warps(Zp << P) + 5, own = warps(Z * (Z - 1) / 2) + warps(Z) + 5 + 1;
    const int diag = warps(A * (A - 1) / 2) + warps(A) + 5 + std::max(pn, own) + 1;
    F.tol_one = std::ldexp((float)one, 4 - 48);
    F.tol_diag = std::ldexp((float)diag, 4 - 48);
}

}  // namespace

namespace {

// fn(first set, sets, values of an entry) for the passes of a fill of K sets
template <class Fn>
int over_passes(int K, Fn &&fn)
{
    const int kv = K == 1 ? 1 : K == 2 ? 2 : 4;
    int rc = CIH_OK;
    for (int k0 = 0; k0 < K && !rc; k0 += kv) {
        const int ks = std::min(kv, K - k0);
        rc = fn(k0, ks, ks == 1 ? 1 : ks == 2 ? 2 : 4);
    }
    return rc;
}

}  // namespace

size_t fill_work_floats(const cih_basis &b, int K)
{
    size_t n = 0;
    if (!fill_splits(b, K)) return 0;
    over_passes(K, [&](int, int, int v) { n += work_floats(b, v); return CIH_OK; });
    return n;
}

int fill_prepare(const cih_basis &b, int K, double hw, const float *tbme, const double *esp, const double *t1, float *work,
                 cudaStream_t st)
{
    FillArgs F{};
    F.K = K;
    F.hw = hw;
    F.tbme = tbme;
    F.tb_sk = b.layout.total;
    F.tb_si = 1;
    F.esp = esp;
    F.t1 = t1;
    return over_passes(K, [&](int k0, int ks, int v) {
        const int rc = launch_prep(b, v, F, work_at(b, work, v, k0, ks), st);
        work += work_floats(b, v);
        return rc;
    });
}

// Whether the stream is being captured: a graph with an allocation in it could not be a
// child graph nor be instantiated twice, so a captured fill takes no scratch (the row
// kernel, the same bits).
static bool capturing(cudaStream_t st)
{
    cudaStreamCaptureStatus s = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(st, &s) == cudaSuccess) return s != cudaStreamCaptureStatusNone;
    (void)cudaGetLastError();
    return true;
}

int launch_fill(const cih_basis &b, const int64_t *rowptr, int K, double hw, const float *tbme, bool interleaved,
                bool em, const double *esp, int32_t *col, float *val, cudaStream_t st, int64_t r0, int64_t r1,
                bool sharded, const double *t1, const float *work, bool prepare)
{
    const int vec4 = interleaved && K % 4 == 0 && ((uintptr_t)tbme & 15) == 0 && (!em || ((uintptr_t)val & 15) == 0);
    FillArgs F{K, hw, tbme, interleaved ? 1 : b.layout.total, interleaved ? (int64_t)K : 1, vec4, em && K > 1 ? 1 : 0,
               esp, col, val, sharded ? 1 : 0, r0, t1, 0.f, 0.f};
    const bool split = fill_splits(b, K);
    if (split) split_tolerances(b, F);
    const int64_t rend = r1 < 0 ? b.dim : r1;
    if (split && work && rend > r0)
        return over_passes(K, [&](int k0, int ks, int v) {
            const FillWork W = work_at(b, const_cast<float *>(work), v, k0, ks);
            work += work_floats(b, v);
            return launch_fill1(b, v, rowptr, F, W, st, false, r0, rend);
        });
    if (split && !work && prepare && copy_pays(b, K, rend - r0) && !capturing(st)) {
        float *own = nullptr;
        const size_t bytes = work_floats(b, K == 1 ? 1 : K == 2 ? 2 : 4) * sizeof(float);        // of the largest pass
        if (cudaMallocFromPoolAsync((void **)&own, bytes, b.pool, st) == cudaSuccess) {
            const int rc = over_passes(K, [&](int k0, int ks, int v) {
                const FillWork W = work_at(b, own, v, k0, ks);
                const int r = launch_prep(b, v, F, W, st);
                return r ? r : launch_fill1(b, v, rowptr, F, W, st, false, r0, rend);
            });
            cudaFreeAsync(own, st);
            return rc;
        }
        (void)cudaGetLastError();
    }
    return launch_rows<1>(b, rowptr, nullptr, F, GradArgs{}, st, false, r0, r1);
}

int prepare_rows(const cih_basis &b, int K)
{
    FillArgs F{};
    F.K = K;
    GradArgs G{};
    G.K = K;
    int rc = launch_rows<0>(b, nullptr, nullptr, F, G, nullptr, true);
    if (!rc) rc = launch_rows<1>(b, nullptr, nullptr, F, G, nullptr, true);
    if (!rc && fill_splits(b, K)) {                          // (a fill without room for its copy)
        FillArgs S = F;
        split_tolerances(b, S);
        rc = launch_rows<1>(b, nullptr, nullptr, S, G, nullptr, true);
    }
    if (!rc) rc = launch_rows<2>(b, nullptr, nullptr, F, G, nullptr, true);
    if (!rc && fill_work_floats(b, K) > 0)
        rc = over_passes(K, [&](int, int, int v) { return launch_fill1(b, v, nullptr, F, FillWork{}, nullptr, true, 0, 0); });
    return rc;
}

int launch_interleave(int K, int64_t len, const float *in, float *out, cudaStream_t st)
{
    if (len * K == 0) return CIH_OK;
    const int blocks = (int)std::min<int64_t>((len * K + 255) / 256, 152 * 16);
    count_launches(1);
    k_interleave<<<blocks, 256, 0, st>>>(K, len, in, out);
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? CIH_OK : cuda_fail(e, "interleave");
}

// psi_fix[i] = psi[i] * 2^61 rounded; |psi| >= 4 cannot be held and sets status
// bit 32.  Grid (blocks, K); part[k * gridDim.x + block] = this block's share of
// ||psi_k||^2.
__global__ void __launch_bounds__(256) k_psi_fix(int64_t dim, const double *psi, long long *psi_fix, double *part, int *status)
{
    __shared__ double red[8];
    const double *v = psi + (int64_t)blockIdx.y * dim;
    long long *o = psi_fix + (int64_t)blockIdx.y * dim;
    double s = 0.0;
    for (int64_t i = blockIdx.x * 256ll + threadIdx.x; i < dim; i += gridDim.x * 256ll) {
        const double x = v[i];
        s += x * x;
        if (!(fabs(x) < 4.0)) {
            atomicOr(status, 32);
            o[i] = 0;
        } else {
            o[i] = __double2ll_rn(x * kPsiScale);
        }
    }
    for (int d = 16; d > 0; d >>= 1) s += __shfl_xor_sync(0xffffffffu, s, d);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < 8; ++w) s += red[w];
        part[(int64_t)blockIdx.y * gridDim.x + blockIdx.x] = s;
    }
}

// ||psi_k||^2 above 1 + 1e-6 sets status bit 32 (|g_t| <= 2 ||psi||^2 must stay
// below the 2^7 the 2^-56 accumulators hold); one warp per set
__global__ void k_psi_norm(int parts, const double *part, int *status)
{
    double s = 0.0;
    for (int i = threadIdx.x; i < parts; i += 32) s += part[(int64_t)blockIdx.x * parts + i];
    for (int d = 16; d > 0; d >>= 1) s += __shfl_xor_sync(0xffffffffu, s, d);
    if (threadIdx.x == 0 && !(s <= 1.0 + 1e-6)) atomicOr(status, 32);
}

namespace {

template <int WARPS>
int launch_grad1_w(const cih_basis &b, const long long *psi, unsigned long long *acc, cudaStream_t st)
{
    const size_t smem = (size_t)f1::S<WARPS> + ((size_t)b.dev.sp[0].n_orb * b.dev.pn_T * 2 + 15) / 16 * 16;
    int dev = 0, sms = 148;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaError_t e = raise_smem_limit((const void *)k_grad1<WARPS>, dev, (int)smem);
    if (e != cudaSuccess) return cuda_fail(e, "adjoint shared memory");
    int per_sm = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_grad1<WARPS>, WARPS * 32, smem);
    per_sm = std::max(per_sm, 1);
    if (b.launch_ctas > 0) per_sm = std::min(per_sm, b.launch_ctas);
    const int64_t want = (b.dim + WARPS - 1) / WARPS;
    count_launches(1);
    k_grad1<WARPS><<<(int)std::min<int64_t>((int64_t)sms * per_sm, want), WARPS * 32, smem, st>>>(b.dev, psi, acc);
    e = cudaGetLastError();
    return e == cudaSuccess ? CIH_OK : cuda_fail(e, "adjoint launch");
}

}  // namespace

size_t grad_pairs_bytes(const cih_basis &b)
{
    if (b.dim < kGradPairsMin || !fill1_fits(b, 1)) return 0;
    const DevBasis &D = b.dev;
    const int64_t np = b.s[0].n_sd, nn = b.s[1].n_sd;
    // 8-byte arrays: neutron-major vector, neutron run starts, proton counts, scan
    // scratch, pn squares; then 4-byte: first partners and level counts
    return 8 * (size_t)(b.dim + (nn + 1) + np + scan_scratch_needed(nn) + b.sq_total) +
           4 * (size_t)(np * (1 + D.sp[0].NL) + nn * (1 + D.sp[1].NL));
}

namespace {

// one vector in the form of k_grad_pairs + k_grad1; 1: not this form (few rows, no
// memory for its scratch, or a shape outside k_grad1's)
int launch_grad1(const cih_basis &b, const long long *fix, unsigned long long *acc, cudaStream_t st)
{
    const size_t bytes = grad_pairs_bytes(b);
    if (bytes == 0) return 1;
    const DevBasis &D = b.dev;
    const int64_t np = b.s[0].n_sd, nn = b.s[1].n_sd, ns = scan_scratch_needed(nn);
    int64_t *buf = nullptr;
    if (cudaMallocFromPoolAsync((void **)&buf, bytes, b.pool, st) != cudaSuccess) {
        (void)cudaGetLastError();
        return 1;
    }
    long long *psin = reinterpret_cast<long long *>(buf);
    int64_t *basen = buf + b.dim, *cntp = basen + nn + 1, *scan = cntp + np;
    unsigned long long *sq = reinterpret_cast<unsigned long long *>(scan + ns);
    int32_t *begp = reinterpret_cast<int32_t *>(sq + b.sq_total), *levp = begp + np, *begn = levp + np * D.sp[0].NL, *levn = begn + nn;
    count_launches(4);
    k_partners<<<(int)((np + 127) / 128), 128, 0, st>>>(D, b.sbuild[0], b.sbuild[1], 0, b.space.twoM, begp, levp, cntp);
    k_partners<<<(int)((nn + 127) / 128), 128, 0, st>>>(D, b.sbuild[0], b.sbuild[1], 1, b.space.twoM, begn, levn, basen);
    int rc = exclusive_scan_i64(basen, nn, scan, ns, st);
    if (!rc) {
        k_psi_neutron_major<<<(int)std::min<int64_t>((b.dim + 255) / 256, 152 * 16), 256, 0, st>>>(D, begn, basen, fix, psin);
        const Partners Pt{{begp, begn}, {levp, levn}, {D.rowbase, basen}, {fix, psin}};
        k_grad_pairs<<<(int)std::min<int64_t>(np + nn, 152 * 32), 256, 0, st>>>(D, Pt, acc, b.dev_status);
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) rc = cuda_fail(e, "adjoint pairs");
    }
    cudaMemsetAsync(sq, 0, sizeof(unsigned long long) * b.sq_total, st);
    if (!rc) rc = b.launch_warps == 8 ? launch_grad1_w<8>(b, fix, sq, st) : launch_grad1_w<16>(b, fix, sq, st);
    if (!rc && b.dev.n_sqrow > 0) {
        count_launches(1);
        k_grad_fold<<<std::min((b.dev.n_sqrow + 7) / 8, 152 * 16), 256, 0, st>>>(D, sq, acc);
    }
    cudaFreeAsync(buf, st);
    return rc;
}

}  // namespace

int launch_grad(const cih_basis &b, const int64_t *rowptr, int K, const double *psi,
                unsigned long long *acc, cudaStream_t st, bool pairs)
{
    const int64_t n = (int64_t)K * b.dim;
    if (n == 0) return CIH_OK;
    const int parts = (int)std::max<int64_t>(1, std::min<int64_t>((b.dim + 1023) / 1024, 152 * 8));
    long long *fix = nullptr;
    cudaError_t e = cudaMallocFromPoolAsync((void **)&fix, sizeof(long long) * n + sizeof(double) * (size_t)parts * K, b.pool, st);
    if (e != cudaSuccess) {
        (void)cudaGetLastError();
        return fail(CIH_ERR_NOMEM, "adjoint: fixed-point vector");
    }
    double *part = reinterpret_cast<double *>(fix + n);
    count_launches(2);
    for (int k0 = 0; k0 < K; k0 += 32768) {                  // (grid.y is limited)
        const int kc = std::min(K - k0, 32768);
        k_psi_fix<<<dim3(parts, kc), 256, 0, st>>>(b.dim, psi + (int64_t)k0 * b.dim, fix + (int64_t)k0 * b.dim,
                                                   part + (int64_t)k0 * parts, b.dev_status);
    }
    k_psi_norm<<<K, 32, 0, st>>>(parts, part, b.dev_status);
    int rc = K == 1 && pairs ? launch_grad1(b, fix, acc, st) : 1;
    if (rc == 1) {
        const GradArgs G{K, fix, acc};
        rc = launch_rows<2>(b, rowptr, nullptr, FillArgs{}, G, st);
    }
    cudaFreeAsync(fix, st);
    return rc;
}

int launch_grad_finish(int64_t n, const unsigned long long *acc, double *grad, cudaStream_t st)
{
    if (n == 0) return CIH_OK;
    int blocks = (int)std::min<int64_t>((n + 255) / 256, 65535);
    count_launches(1);
    k_fix_to_double<<<blocks, 256, 0, st>>>(n, acc, grad);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(e, "gradient finish");
    return CIH_OK;
}

}  // namespace cih
