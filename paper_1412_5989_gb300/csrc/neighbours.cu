// Device set-up of a basis: upload the host tables and build, per species,
// the neighbour lists the Hamiltonian kernels walk.
//
// Sec. 4.1 of the paper locates nonzeros either by testing every element of
// a dense block or, for sparse blocks, by iterating only over the quantum
// number combinations that can be nonzero.  Both appear here, one level
// down: the same-class forward list of a sub-determinant is found by testing
// every later member of its (2M, parity) class (XOR + popcount), and the
// one-move list by generating each single-orbital move and looking the result
// up in the sorted sub-determinant table.  Sec. 5.2's lesson (build index
// structures contiguously, one allocation each) applies to every list.
#include <algorithm>
#include <cstring>

#include <functional>
#include <mutex>
#include <type_traits>

#include "cih_internal.h"

namespace cih {
namespace {



// (base is 256-byte aligned: strings of two and four words load 16 bytes at a time)
template <int W>
__device__ __forceinline__ void load_bits(const uint64_t *base, int64_t i, uint64_t (&o)[W])
{
    if constexpr (W == 1) {
        o[0] = __ldg(base + i);
    } else {
        const ulonglong2 *b = reinterpret_cast<const ulonglong2 *>(base) + i * (W / 2);
#pragma unroll
        for (int w = 0; w < W / 2; ++w) {
            const ulonglong2 v = __ldg(b + w);
            o[2 * w] = v.x;
            o[2 * w + 1] = v.y;
        }
    }
}

template <int W>
__device__ __forceinline__ uint32_t hash_bits(const uint64_t *b)
{
    uint64_t h = 0x9E3779B97F4A7C15ull;
#pragma unroll
    for (int w = 0; w < W; ++w) {
        h ^= b[w] + 0x632BE59BD9B4E019ull + (h << 6) + (h >> 2);
        h *= 0xBF58476D1CE4E5B9ull;
    }
    return (uint32_t)(h ^ (h >> 31));
}

// insert every sub-det index (all keys distinct: claim the first empty slot)
template <int W>
__global__ void k_hash_build(SpeciesBuild S, int32_t *table)
{
    for (int64_t x = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; x < S.n_sd; x += (int64_t)gridDim.x * blockDim.x) {
        uint32_t h = hash_bits<W>(S.bits + x * W) & S.hash_mask;
        for (uint32_t probe = 0; probe <= S.hash_mask; ++probe) {
            if (atomicCAS(&table[h], -1, (int32_t)x) == -1) break;
            h = (h + 1) & S.hash_mask;
        }
    }
}

// index of the sub-det with bits `yb`, or -1 (hash lookup; at most capacity probes)
template <int W>
__device__ int find_subdet(const SpeciesBuild &S, const uint64_t (&yb)[W])
{
    uint32_t h = hash_bits<W>(yb) & S.hash_mask;
    for (uint32_t probe = 0; probe <= S.hash_mask; ++probe) {
        const int32_t x = S.hash[h];
        if (x < 0) return -1;
        uint64_t xb[W];
        load_bits<W>(S.bits, x, xb);
        bool eq = true;
#pragma unroll
        for (int w = 0; w < W; ++w) eq &= xb[w] == yb[w];
        if (eq) return x;
        h = (h + 1) & S.hash_mask;
    }
    return -1;
}

// bit k of a string, and the string with bit k flipped (word selects instead of
// indexed words, which would put the string into local memory)
template <int W>
__device__ __forceinline__ bool has_bit(const uint64_t (&x)[W], int k)
{
    uint64_t v = 0;
#pragma unroll
    for (int w = 0; w < W; ++w) v = w == (k >> 6) ? x[w] : v;
    return (v >> (k & 63)) & 1;
}

template <int W>
__device__ __forceinline__ void flip_bit(uint64_t (&x)[W], int k)
{
#pragma unroll
    for (int w = 0; w < W; ++w) x[w] ^= w == (k >> 6) ? 1ull << (k & 63) : 0ull;
}

template <int W>
__device__ __forceinline__ int low_bit(const uint64_t (&x)[W])
{
#pragma unroll
    for (int w = 0; w < W; ++w)
        if (x[w]) return w * 64 + __ffsll((long long)x[w]) - 1;
    return -1;
}

template <int W>
__device__ __forceinline__ int count_below(const uint64_t (&R)[W], int k)
{
    int c = 0;
#pragma unroll
    for (int w = 0; w < W; ++w) {
        int lo = w * 64;
        if (k >= lo + 64) c += __popcll(R[w]);
        else if (k > lo) c += __popcll(R[w] & ((1ull << (k - lo)) - 1));
    }
    return c;
}

// Neutron one-move lists packed, bra x -> ket y (DevBasis::n1p): b = orbital
// in x only, d = orbital in y only, R = common orbitals, sign (-1)^(#R below b
// + #R below d); orbs[b] = r(b) | t(b) << 8.
template <int W>
__global__ void k_n1_pack(SpeciesBuild S, const int64_t *off, const int32_t *list, const uint16_t *orbs, int2 *packed)
{
    int lane = threadIdx.x & 31;
    int64_t warp = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t x = warp; x < S.n_sd; x += nwarps) {
        uint64_t bx[W];
        load_bits<W>(S.bits, x, bx);
        for (int64_t t = off[x] + lane; t < off[x + 1]; t += 32) {
            uint64_t by[W], R[W], dx[W], dy[W];
            const int y = list[t];
            load_bits<W>(S.bits, y, by);
#pragma unroll
            for (int w = 0; w < W; ++w) { R[w] = bx[w] & by[w]; dx[w] = bx[w] & ~by[w]; dy[w] = by[w] & ~bx[w]; }
            const int b = low_bit<W>(dx), d = low_bit<W>(dy);
            const uint32_t sg = (count_below<W>(R, b) + count_below<W>(R, d)) & 1, ob = orbs[b], od = orbs[d];
            packed[t] = make_int2(y, (int)((od & 0xFF) | (ob & 0xFF) << 8 | (ob >> 8) << 16 | (od >> 8) << 21 | sg << 26));
        }
    }
}

// Splits the staged forward list of each sub-det x (one warp each) into its
// two-moves, ascending from the slot's start, and its one-moves, ascending from
// the slot's end backwards (DevSpecies::fw_rec, fw_tb), and counts the
// two-moves per level.  A two-move's table index (<< 1) and sign bit: bra x ->
// ket y, orbitals offset by `base` into the pair table; a one-move is stored
// as ~(b | d << 8 | sign << 16) with b in x only, d in y only.  rowbase / nb:
// the record holds the column base of y (protons), or null: y itself.
template <int W>
__global__ void k_split(SpeciesBuild S, int base, int N0, int NL, const int32_t *cls_of, const int64_t *class_stage,
                        const int64_t *off, const int32_t *stage, const int64_t *rowbase, const int32_t *nb,
                        const int32_t *pid, const int32_t *gsize, const int64_t *goff, int ntot, int2 *rec, int32_t *tb,
                        int32_t *lev, int *status)
{
    const int lane = threadIdx.x & 31;
    const unsigned lt = (1u << lane) - 1;
    const int64_t warp = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t x = warp; x < S.n_sd; x += nwarps) {
        uint64_t bx[W];
        load_bits<W>(S.bits, x, bx);
        const int c = cls_of[x];
        const int64_t cb = S.cls_begin[c], m = S.cls_endc[c] - cb, r = x - cb;
        const int32_t *in = stage + class_stage[c] + r * (m - 1) - r * (r - 1) / 2;
        const int64_t o0 = off[x], o1 = off[x + 1];
        const int len = (int)(o1 - o0);
        int n2 = 0, n1 = 0;                                    // two- and one-moves so far
        int at_lev = 0;                                        // lane l: two-moves at levels <= l
        for (int t0 = 0; t0 < len; t0 += 32) {
            const bool on = t0 + lane < len;
            const int y = on ? in[t0 + lane] : (int)x;
            uint64_t by[W], R[W], dx[W], dy[W];
            load_bits<W>(S.bits, y, by);
            int pc = 0;
#pragma unroll
            for (int w = 0; w < W; ++w) {
                R[w] = bx[w] & by[w]; dx[w] = bx[w] & ~by[w]; dy[w] = by[w] & ~bx[w];
                pc += __popcll(dx[w]);
            }
            const bool two = on && pc == 2, one = on && pc != 2;
            const unsigned m2 = __ballot_sync(0xffffffffu, two), m1 = __ballot_sync(0xffffffffu, one);
            const int lv = (S.N[y] - N0) >> 1;
            for (int l = 0; l < NL; ++l) {
                const unsigned ml = __ballot_sync(0xffffffffu, two && lv <= l);
                if (lane == l) at_lev += __popc(ml);
            }
            if (on) {
                const int k2 = n2 + __popc(m2 & lt), k1 = n1 + __popc(m1 & lt);
                const int64_t slot = two ? o0 + k2 : o1 - 1 - k1;
                rec[slot] = make_int2(rowbase ? (int)(rowbase[y] - nb[y]) : y, (two ? k1 : k2) | lv << 24);
                if (one) {
                    const int b1 = low_bit<W>(dx), d1 = low_bit<W>(dy);
                    const int s1 = (count_below<W>(R, b1) + count_below<W>(R, d1)) & 1;
                    tb[slot] = ~(int32_t)(b1 | (d1 << 8) | (s1 << 16));
                } else {
                    const int a1 = low_bit<W>(dx), c1 = low_bit<W>(dy);
                    flip_bit<W>(dx, a1);
                    flip_bit<W>(dy, c1);
                    const int a2 = low_bit<W>(dx), c2 = low_bit<W>(dy);
                    int sg = (count_below<W>(R, a1) + count_below<W>(R, a2) + count_below<W>(R, c1) + count_below<W>(R, c2)) & 1;
                    int32_t e1 = pid[(base + a1) * ntot + base + a2], e2 = pid[(base + c1) * ntot + base + c2];
                    if (e1 < 0 || e2 < 0 || ((e1 ^ e2) & (0xFFF << 16))) {
                        atomicOr(status, 4);
                        tb[slot] = 0;
                    } else {
                        int g = (e1 >> 16) & 0xFFF;
                        int64_t u = e1 & 0xFFFF, v = e2 & 0xFFFF;
                        if (u > v) { int64_t q = u; u = v; v = q; }
                        int64_t n = gsize[g];
                        int64_t idx = goff[g] + u * n - u * (u - 1) / 2 + (v - u);
                        tb[slot] = (int32_t)((idx << 1) | sg);
                    }
                }
            }
            n2 += __popc(m2);
            n1 += __popc(m1);
        }
        if (lane < NL) lev[x * NL + lane] = at_lev;
    }
}

// one-move entries of each sub-det below itself
__global__ void k_n1_self(int64_t n, const int64_t *n1_off, const int32_t *n1, int32_t *self)
{
    for (int64_t x = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; x < n; x += (int64_t)gridDim.x * blockDim.x) {
        int64_t lo = n1_off[x], hi = n1_off[x + 1];
        const int64_t a0 = lo;
        while (lo < hi) {
            const int64_t mid = (lo + hi) >> 1;
            if (n1[mid] < x) lo = mid + 1; else hi = mid;
        }
        self[x] = (int32_t)(lo - a0);
    }
}

// Group records of each proton sub-det (DevBasis::grp), one warp per p.  PASS
// 0 counts them; PASS 1 writes them, and the packed one-moves (DevBasis::l1).
template <int W, int PASS>
__global__ void k_groups(SpeciesBuild S, DevBasis B, int64_t *gcnt, int4 *grp, int2 *l1)
{
    const DevSpecies &SP = B.sp[0], &SN = B.sp[1];
    const int lane = threadIdx.x & 31;
    const unsigned lt = (1u << lane) - 1;
    const int64_t warp = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    const int NL = SP.NL;
    for (int64_t p = warp; p < S.n_sd; p += nwarps) {
        const int64_t i0 = SP.n1_off[p] + SP.n1_self[p], i1 = SP.n1_off[p + 1];
        const int cend = SP.cls_end[p];
        int64_t mid = i0, hi = i1;                              // first one-move beyond p's class
        while (mid < hi) {
            const int64_t h = (mid + hi) >> 1;
            if (SP.n1[h] < cend) mid = h + 1; else hi = h;
        }
        const int64_t later = mid;
        // directory positions of the segment of q's range in the list of a row neutron of p
        auto seg = [&](int q) {
            const int Lq = B.Nlim - S.N[q], dM = S.M2[p] - S.M2[q];
            if (dM > B.DM || dM < -B.DM || Lq < SN.N0) return 0;       // no neutron one-move reaches it
            const int rc = ((dM + B.DM) >> 1) * 2 + (Lq & 1), l = min((Lq - SN.N0) >> 1, SN.NL - 1);
            return rc * SN.NL | (1 + rc * SN.NL + l) << 16;
        };
        // own class: lane l holds level l
        const int par = (S.N[p] - SP.N0) & 1;
        int t2 = lane < NL ? SP.fw_lev[p * NL + lane] : 0, e = (int)(later - i0);
        if (lane < NL) {                                        // one-moves of levels <= lane
            int64_t lo = i0, h2 = later;
            while (lo < h2) {
                const int64_t h = (lo + h2) >> 1;
                if (((S.N[SP.n1[h]] - SP.N0) >> 1) <= lane) lo = h + 1; else h2 = h;
            }
            e = (int)(lo - i0);
        }
        const int pe = __shfl_up_sync(0xffffffffu, e, 1), pt2 = __shfl_up_sync(0xffffffffu, t2, 1);
        const int e0 = lane ? pe : 0, t20 = lane ? pt2 : 0;
        const bool has = lane < NL && (e > e0 || t2 > t20);
        const unsigned hm = __ballot_sync(0xffffffffu, has);
        const int64_t g0 = PASS ? gcnt[p] : 0;
        if (PASS == 1 && has) {
            const int Nq = SP.N0 + 2 * lane + par, Lq = B.Nlim - Nq;
            int st = 0;
            if (Lq >= SN.N0) {
                const int rc = (B.DM >> 1) * 2 + (Lq & 1), l = min((Lq - SN.N0) >> 1, SN.NL - 1);
                st = rc * SN.NL | (1 + rc * SN.NL + l) << 16;
            }
            grp[g0 + __popc(hm & lt)] = make_int4(e0 | (e - e0) << 16, st, t2 - t20, (1 + Lq) | t20 << 8);
        }
        int ng = __popc(hm);
        const int gl = ng;                                      // first later-class group
        for (int64_t t0 = later; t0 < i1; t0 += 32) {
            const int64_t t = t0 + lane;
            const int q = t < i1 ? SP.n1[t] : 0;
            const int b = t > later && t < i1 ? SP.n1[t - 1] : -1;
            const bool first = t < i1 && (b < 0 || SP.cls_end[q] != SP.cls_end[b] || S.N[q] != S.N[b]);
            const unsigned fm = __ballot_sync(0xffffffffu, first);
            if (PASS == 1 && first) grp[g0 + ng + __popc(fm & lt)] = make_int4((int)(t - i0), seg(q), 0, 0);
            ng += __popc(fm);
        }
        if (PASS == 0) {
            if (lane == 0) gcnt[p] = ng;
            continue;
        }
        __syncwarp();
        for (int j0 = gl; j0 < ng; j0 += 32) {                  // members of the later-class groups
            const int j = j0 + lane;
            int a = 0, z = 0;
            if (j < ng) {
                a = grp[g0 + j].x & 0xFFFF;
                z = j + 1 < ng ? grp[g0 + j + 1].x & 0xFFFF : (int)(i1 - i0);
            }
            __syncwarp();
            if (j < ng) grp[g0 + j].x = a | (z - a) << 16;
            __syncwarp();
        }
        uint64_t pb[W];
        load_bits<W>(S.bits, p, pb);
        for (int64_t t = i0 + lane; t < i1; t += 32) {
            const int q = SP.n1[t];
            uint64_t qb[W], R[W], dx[W], dy[W];
            load_bits<W>(S.bits, q, qb);
#pragma unroll
            for (int w = 0; w < W; ++w) { R[w] = pb[w] & qb[w]; dx[w] = pb[w] & ~qb[w]; dy[w] = qb[w] & ~pb[w]; }
            const int a = low_bit<W>(dx), c = low_bit<W>(dy);
            const int sg = (count_below<W>(R, a) + count_below<W>(R, c)) & 1;
            l1[t] = make_int2((int)(B.rowbase[q] - B.nb[q]), a | c << 8 | sg << 16 | B.pn_a[a] << 17);
        }
    }
}

// occupied orbitals of each sub-det, ascending, and the move codes of each
// orbital kept (codes[a]: DevBasis::occ_code)
template <int W>
__global__ void k_occ(SpeciesBuild S, int Z, const int32_t *codes, uint8_t *occ, int32_t *occ_code)
{
    for (int64_t x = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; x < S.n_sd; x += (int64_t)gridDim.x * blockDim.x) {
        int k = 0;
        for (int w = 0; w < W; ++w) {
            uint64_t m = S.bits[x * W + w];
            while (m) {
                const int a = w * 64 + __ffsll((long long)m) - 1;
                occ[x * Z + k] = (uint8_t)a;
                occ_code[x * Z + k++] = codes[a];
                m &= m - 1;
            }
        }
    }
}

// bucket directory of each neutron one-move list (DevBasis::dir)
__global__ void k_dir(SpeciesBuild S, const int64_t *off, const int32_t *list, int N0, int NL, int DM, int dir_len,
                      int16_t *dir)
{
    int lane = threadIdx.x & 31;
    int64_t warp = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t x = warp; x < S.n_sd; x += nwarps) {
        const int64_t a0 = off[x], a1 = off[x + 1];
        const int M0 = S.M2[x];
        int16_t *d = dir + x * (int64_t)dir_len;
        if (lane == 0) d[0] = 0;
        for (int b = lane; b < dir_len - 1; b += 32) {
            // entries with bucket key <= b: keys are non-decreasing along the sorted list
            int64_t lo = a0, hi = a1;
            while (lo < hi) {
                const int64_t mid = (lo + hi) >> 1;
                const int y = list[mid];
                const int key = ((((int)S.M2[y] - M0 + DM) >> 1) * 2 + (S.N[y] & 1)) * NL + ((S.N[y] - N0) >> 1);
                if (key <= b) lo = mid + 1; else hi = mid;
            }
            d[1 + b] = (int16_t)(lo - a0);
        }
    }
}

// per-sub-det records of the row kernels
__global__ void k_proton_rec(DevBasis B, const int64_t *goff, ProtonRec *rec)
{
    const DevSpecies &SP = B.sp[0], &SN = B.sp[1];
    for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < SP.n_sd; p += (int64_t)gridDim.x * blockDim.x) {
        const int Lp = B.Nlim - SP.N[p], l = min((Lp - SN.N0) >> 1, SN.NL - 1);
        ProtonRec r;
        r.l1 = SP.n1_off[p] + SP.n1_self[p];
        r.fw = SP.fw_off[p];
        r.g0 = goff[p];
        r.fwlen = (int32_t)(SP.fw_off[p + 1] - r.fw);
        r.colb = (int32_t)(B.rowbase[p] - B.nb[p]);
        r.nb = B.nb[p];
        r.ng = (int32_t)(goff[p + 1] - r.g0);
        r.dirA = 1 + ((B.DM >> 1) * 2 + (Lp & 1)) * SN.NL + l;
        r.levA = l;
        rec[p] = r;
    }
}

__global__ void k_neutron_rec(DevSpecies SN, NeutronRec *rec)
{
    for (int64_t n = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; n < SN.n_sd; n += (int64_t)gridDim.x * blockDim.x)
        rec[n] = NeutronRec{SN.n1_off[n], SN.fw_off[n], (int32_t)(SN.fw_off[n + 1] - SN.fw_off[n]), SN.n1_self[n], SN.N[n], 0};
}

// row -> proton sub-det, and (walk not null) the order the one-set kernels take
// the rows in: inside each aligned run of kWalkRun proton sub-dets those with the
// same neutron range go side by side, n by n.  One warp per p.
__global__ void k_row_p(int64_t np, const int64_t *rowbase, const int32_t *nb, const int32_t *nc, int32_t *row_p, int2 *walk)
{
    int lane = threadIdx.x & 31;
    int64_t warp = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t p = warp; p < np; p += nwarps) {
        const int64_t r0 = rowbase[p], r1 = rowbase[p + 1];
        for (int64_t r = r0 + lane; r < r1; r += 32) row_p[r] = (int32_t)p;
        if (!walk) continue;
        int64_t g0 = p, g1 = p + 1;                            // p's neighbours in the run with its range
        while (g0 > p / kWalkRun * kWalkRun && nb[g0 - 1] == nb[p] && nc[g0 - 1] == nc[p]) --g0;
        while (g1 < np && g1 < (p / kWalkRun + 1) * kWalkRun && nb[g1] == nb[p] && nc[g1] == nc[p]) ++g1;
        for (int64_t r = r0 + lane; r < r1; r += 32)
            walk[rowbase[g0] + (r - r0) * (g1 - g0) + (p - g0)] = make_int2((int)p, (int)r);
    }
}

// Single-pass forward lists: sub-det x at rank r of a class [cb, ce) of size
// m has room for m - r - 1 entries at stage offset
//   class_stage[c] + r (m - 1) - r (r - 1) / 2,
// written in ascending order; cnt[x] gets the count.  One warp per sub-det, lanes
// over the later class members.  Strings of several words are first compared by
// their words' exclusive or (S.fold): folding can only lower the count of
// differing bits, so what it rejects (most) needs no full comparison; the rest
// queues up in shared memory and is compared in full 32 at a time.  Bound by
// the instructions of the comparisons: 288 us for a species of 4+4 Nmax=6 with
// two words compared for every member, 192 us with one.
template <int W>
__global__ void __launch_bounds__(256) k_forward_staged(SpeciesBuild S, const int32_t *cls_of, const int64_t *class_stage, int64_t *cnt,
                                                        int32_t *stage)
{
    __shared__ int32_t queue[8][64];
    const int lane = threadIdx.x & 31;
    const unsigned lt = (1u << lane) - 1;
    int32_t *q = queue[threadIdx.x >> 5];
    int64_t warp = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t x = warp; x < S.n_sd; x += nwarps) {
        uint64_t bx[W];
        load_bits<W>(S.bits, x, bx);
        uint64_t fx = 0;
#pragma unroll
        for (int w = 0; w < W; ++w) fx ^= bx[w];
        const int c = cls_of[x];
        const int64_t cb = S.cls_begin[c], m = S.cls_endc[c] - cb, r = x - cb;
        int32_t *out = stage + class_stage[c] + r * (m - 1) - r * (r - 1) / 2;
        const int end = S.cls_end[x];
        int64_t pos = 0;
        int nq = 0;
        auto compare = [&](int n) {                            // the first n queued members
            bool hit = false;
            int y = 0;
            if (lane < n) {
                y = q[lane];
                uint64_t by[W];
                load_bits<W>(S.bits, y, by);
                int d = 0;
#pragma unroll
                for (int w = 0; w < W; ++w) d += __popcll(bx[w] ^ by[w]);
                hit = d <= 4;
            }
            const unsigned msk = __ballot_sync(0xffffffffu, hit);
            if (hit) out[pos + __popc(msk & lt)] = y;
            pos += __popc(msk);
        };
#pragma unroll 2
        for (int y0 = (int)x + 1; y0 < end; y0 += 32) {
            const int y = y0 + lane;
            const bool near = y < end && __popcll(fx ^ (W == 1 ? __ldg(S.bits + y) : __ldg(S.fold + y))) <= 4;
            const unsigned msk = __ballot_sync(0xffffffffu, near);
            if (W == 1) {                                      // the fold is the string
                if (near) out[pos + __popc(msk & lt)] = y;
                pos += __popc(msk);
                continue;
            }
            if (near) q[nq + __popc(msk & lt)] = y;
            nq += __popc(msk);
            __syncwarp();
            if (nq >= 32) {
                compare(32);
                nq -= 32;
                __syncwarp();
                const int32_t k = lane < nq ? q[32 + lane] : 0;
                __syncwarp();
                if (lane < nq) q[lane] = k;
                __syncwarp();
            }
        }
        if (nq > 0) compare(nq);
        if (lane == 0) cnt[x] = pos;
        __syncwarp();
    }
}

// fold[x] = exclusive or of the words of x's bit string
__global__ void k_fold(int64_t n, int W, const uint64_t *bits, uint64_t *fold)
{
    for (int64_t x = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; x < n; x += (int64_t)gridDim.x * blockDim.x) {
        uint64_t f = 0;
        for (int w = 0; w < W; ++w) f ^= bits[x * W + w];
        fold[x] = f;
    }
}

// Single-pass one-move lists: each sub-det writes its moves (unsorted) into
// a slot of `cap` entries; cnt[x] gets the count.  One warp per sub-det: the
// moves (r, a) whose image has the (2M, N) of some sub-det (S.keep; about one in
// four does) queue up in shared memory, and the hash look-ups, two dependent
// reads each, run for 32 of them at a time: 343 us a species at 4+4 Nmax=6 with a
// look-up for every free target orbital, most lanes idle, 269 us so.
constexpr int kMoveQueue = 64;

template <int W>
__global__ void __launch_bounds__(256) k_onemove_staged(SpeciesBuild S, int cap, int64_t *cnt, int32_t *stage)
{
    __shared__ uint16_t queue[8][kMoveQueue];
    const int lane = threadIdx.x & 31;
    const unsigned lt = (1u << lane) - 1;
    uint16_t *q = queue[threadIdx.x >> 5];
    int64_t warp = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t x = warp; x < S.n_sd; x += nwarps) {
        uint64_t bx[W];
        load_bits<W>(S.bits, x, bx);
        const int Nx = S.N[x], Mx = S.M2[x];
        int32_t *out = stage + x * (int64_t)cap;
        int pos = 0, nq = 0;
        auto look_up = [&](int n) {                            // the first n queued moves
            int found = -1;
            if (lane < n) {
                const int r = q[lane] & 0xFF, a = q[lane] >> 8;
                uint64_t yb[W];
#pragma unroll
                for (int v = 0; v < W; ++v) yb[v] = bx[v];
                flip_bit<W>(yb, r);
                flip_bit<W>(yb, a);
                found = find_subdet<W>(S, yb);
            }
            const unsigned msk = __ballot_sync(0xffffffffu, found >= 0);
            if (found >= 0) out[pos + __popc(msk & lt)] = found;
            pos += __popc(msk);
        };
#pragma unroll
        for (int w = 0; w < W; ++w) {
            uint64_t occ = bx[w];
            while (occ) {
                const int r = w * 64 + __ffsll((long long)occ) - 1;
                occ &= occ - 1;
                const int Nr = S.oN[r], Mr = S.om2[r];
                // targets a with Nx - Nr + N_a <= Nsub_max: a prefix of the shell-ordered orbitals
                const int lim = S.Nsub_max - Nx + Nr;
                const int aend = lim < 0 ? 0 : lim >= S.maxN ? S.n_orb : S.orb_upto[lim];
                for (int a0 = 0; a0 < aend; a0 += 32) {
                    const int a = a0 + lane;
                    bool ok = false;
                    if (a < aend && !has_bit<W>(bx, a)) {
                        const int Ny = Nx - Nr + S.oN[a], k = Mx - Mr + S.om2[a] + S.mtop;
                        ok = Ny >= 0 && Ny <= S.Nsub_max && k >= 0 && k <= 2 * S.mtop && S.keep[k * (S.Nsub_max + 1) + Ny];
                    }
                    const unsigned msk = __ballot_sync(0xffffffffu, ok);
                    if (ok) q[nq + __popc(msk & lt)] = (uint16_t)(r | a << 8);
                    nq += __popc(msk);
                    __syncwarp();
                    if (nq >= 32) {
                        look_up(32);
                        nq -= 32;
                        __syncwarp();
                        const uint16_t m = lane < nq ? q[32 + lane] : 0;
                        __syncwarp();
                        if (lane < nq) q[lane] = m;
                        __syncwarp();
                    }
                }
            }
        }
        if (nq > 0) look_up(nq);
        if (lane == 0) cnt[x] = pos;
        __syncwarp();
    }
}

// the staged moves sorted (ascending), written compact at off[x]: one warp per
// list, bitonic in shared memory (tile entries a warp, a power of two >= cap).  The
// lists have some 100 entries: a block to each waited at its barriers, 280 us a
// species at 4+4 Nmax=6 against 143 us.
__global__ void __launch_bounds__(256) k_onemove_compact_sort(int64_t n, int cap, int tile, const int64_t *off, const int32_t *stage,
                                                              int32_t *out)
{
    extern __shared__ int32_t sort_sh[];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    int32_t *sh = sort_sh + wid * tile;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t x = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5; x < n; x += nw) {
        const int64_t o = off[x];
        const int len = (int)(off[x + 1] - o);
        const int32_t *in = stage + x * (int64_t)cap;
        if (len <= 32) {                          // small lists: place by rank
            const int32_t v = lane < len ? in[lane] : INT32_MAX;
            int rank = 0;
            for (int j = 0; j < len; ++j) rank += __shfl_sync(0xffffffffu, v, j) < v;
            if (lane < len) out[o + rank] = v;
            continue;
        }
        int P = 64;
        while (P < len) P <<= 1;
        for (int i = lane; i < P; i += 32) sh[i] = i < len ? in[i] : INT32_MAX;
        __syncwarp();
        for (int k = 2; k <= P; k <<= 1)
            for (int j = k >> 1; j > 0; j >>= 1) {
                for (int t = lane; t < P / 2; t += 32) {       // pair t: i without bit j, and i | j
                    const int i = ((t & ~(j - 1)) << 1) | (t & (j - 1)), l = i | j;
                    const int32_t a = sh[i], c = sh[l];
                    if ((a > c) == ((i & k) == 0)) { sh[i] = c; sh[l] = a; }
                }
                __syncwarp();
            }
        for (int i = lane; i < len; i += 32) out[o + i] = sh[i];
        __syncwarp();
    }
}

template <class T>
int dev_alloc(cih_basis &b, T **p, size_t n)
{
    *p = nullptr;
    size_t bytes = (std::max<size_t>(n, 1) * sizeof(T) + 255) / 256 * 256;
    cudaError_t e = cudaMallocFromPoolAsync((void **)p, bytes, b.pool, b.stream);
    if (e != cudaSuccess) {
        *p = nullptr;
        (void)cudaGetLastError();
        return fail(CIH_ERR_NOMEM, std::string("device allocation failed: ") + cudaGetErrorString(e));
    }
    b.buffers.owned.push_back((void *)*p);
    return CIH_OK;
}

// return a buffer to the pool once the stream has passed its last use
template <class T>
void dev_free(cih_basis &b, T *p)
{
    if (!p) return;
    auto &v = b.buffers.owned;
    for (size_t i = 0; i < v.size(); ++i)
        if (v[i] == (void *)p) { v.erase(v.begin() + i); break; }
    cudaFreeAsync((void *)p, b.stream);
}

template <class T>
int upload(cih_basis &b, T **p, const std::vector<T> &h, cudaStream_t st)
{
    int rc = dev_alloc(b, p, h.size());
    if (rc) return rc;
    if (!h.empty()) {
        cudaError_t e = cudaMemcpyAsync(*p, h.data(), h.size() * sizeof(T), cudaMemcpyHostToDevice, st);
        if (e != cudaSuccess) return cuda_fail(e, "upload");
    }
    return CIH_OK;
}

// Small host arrays travel to the device together: one allocation and one copy
// for all that are added before flush() (a separate copy of each costs about as
// much host time as a kernel launch; a basis has some forty).  The pointers are
// set by flush(); arrays above kPackMost go by themselves.
struct Packer {
    static constexpr size_t kPackMost = 1 << 16;
    cih_basis &b;
    cudaStream_t st;
    std::vector<unsigned char> host;
    std::vector<std::pair<void **, size_t>> at;
    int rc = CIH_OK;

    Packer(cih_basis &b_, cudaStream_t s) : b(b_), st(s) {}
    template <class T>
    void add(T **p, const std::vector<T> &h)
    {
        if (rc) return;
        if (h.size() * sizeof(T) > kPackMost) {
            rc = upload(b, p, h, st);
            return;
        }
        const size_t o = (host.size() + 255) / 256 * 256;
        host.resize(o + std::max<size_t>(h.size() * sizeof(T), 1));
        if (!h.empty()) std::memcpy(host.data() + o, h.data(), h.size() * sizeof(T));
        at.push_back({(void **)p, o});
    }
    int flush()
    {
        if (rc || at.empty()) return rc;
        unsigned char *d;
        if ((rc = upload(b, &d, host, st))) return rc;
        for (auto &x : at) *x.first = d + x.second;
        at.clear();
        host.clear();
        return CIH_OK;
    }
};

int grid_for(int64_t warps)
{
    int dev = 0, sms = 148;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    int64_t blocks = (warps + 7) / 8;
    return (int)std::max<int64_t>(1, std::min<int64_t>(blocks, (int64_t)sms * 16));
}

// fn(std::integral_constant<int, W>) for the basis' words per bit string
template <class Fn>
void with_words(int W, Fn &&fn)
{
    if (W == 1) fn(std::integral_constant<int, 1>());
    else if (W == 2) fn(std::integral_constant<int, 2>());
    else fn(std::integral_constant<int, 4>());
}

// species t: host arrays (built for both species side by side), then their
// upload and the one-move hash table
struct SpeciesHost {
    std::vector<uint64_t> bits;
    std::vector<int8_t> N, oN;
    std::vector<int16_t> M2, om2;
    std::vector<int32_t> cls_end, cb, ce, cls_of;
    std::vector<int64_t> class_stage;         // staged forward lists: first slot of each class
    int64_t fw_stage = 0;                     // and their total
    std::vector<uint8_t> keep;                // (2M + mtop, N): some sub-det has it
    int mtop = 0;
};

// Neighbour lists of one species, in three phases so that both species'
// kernels queue back to back and the host work in between overlaps them:
//   1. staged forward and one-move passes, their counts scanned, list totals
//      copied to pinned host memory;
//   2. (after one synchronisation) exact-size one-move lists: compaction and sort;
//   3. (once the table layout is on the device) the forward lists split into
//      one- and two-moves, with table indices.
struct Lists {
    int64_t n = 0, ns = 0;
    int64_t *cnt_fw = nullptr, *cnt_n1 = nullptr, *scratch = nullptr, *d_class_stage = nullptr;
    int32_t *d_cls_of = nullptr, *fw_st = nullptr, *n1_st = nullptr, *n1 = nullptr;
    int cap1 = 1, grid = 1;
    int64_t *tot = nullptr;                   // pinned: forward and one-move totals
};

template <int W>
int lists_phase1(cih_basis &b, int t, SpeciesBuild &S, const SpeciesHost &H, Lists &L, cudaStream_t st)
{
    const Species &hs = b.s[t];
    const int64_t n = L.n = S.n_sd;
    int rc;
    if ((rc = dev_alloc(b, &L.cnt_fw, n + 1)) || (rc = dev_alloc(b, &L.cnt_n1, n + 1))) return rc;
    L.ns = scan_scratch_needed(n);
    if ((rc = dev_alloc(b, &L.scratch, L.ns))) return rc;
    L.grid = grid_for(n);
    // staging: forward lists by class triangle, one-move lists by fixed slots
    L.cap1 = std::max(1, hs.Z * std::max(0, hs.n_orb - hs.Z));
    if (L.cap1 > kSortTile) return fail(CIH_ERR_UNSUPPORTED, "one-move lists longer than the sort tile");
    if ((rc = dev_alloc(b, &L.fw_st, H.fw_stage)) || (rc = dev_alloc(b, &L.n1_st, (size_t)n * L.cap1)))
        return rc;
    if (n > 0) {
        count_launches(2);
        k_forward_staged<W><<<L.grid, 256, 0, st>>>(S, L.d_cls_of, L.d_class_stage, L.cnt_fw, L.fw_st);
        k_onemove_staged<W><<<L.grid, 256, 0, st>>>(S, L.cap1, L.cnt_n1, L.n1_st);
    }
    if ((rc = exclusive_scan_i64(L.cnt_fw, n, L.scratch, L.ns, st))) return rc;
    if ((rc = exclusive_scan_i64(L.cnt_n1, n, L.scratch, L.ns, st))) return rc;
    cudaMemcpyAsync(&L.tot[0], L.cnt_fw + n, sizeof(int64_t), cudaMemcpyDeviceToHost, st);
    cudaMemcpyAsync(&L.tot[1], L.cnt_n1 + n, sizeof(int64_t), cudaMemcpyDeviceToHost, st);
    return CIH_OK;
}

int lists_phase2(cih_basis &b, int t, SpeciesBuild &S, Lists &L, cudaStream_t st)
{
    const int64_t n = L.n;
    int rc;
    int32_t *self;
    if ((rc = dev_alloc(b, &L.n1, L.tot[1])) || (rc = dev_alloc(b, &self, n))) return rc;
    if (n > 0) {
        count_launches(2);
        int tile = 64;
        while (tile < L.cap1) tile <<= 1;
        const int wpb = std::min(8, 32768 / tile);              // at most 128 KB of shared memory a block
        const size_t sh = sizeof(int32_t) * (size_t)tile * wpb;
        const cudaError_t e = cudaFuncSetAttribute(k_onemove_compact_sort, cudaFuncAttributeMaxDynamicSharedMemorySize, 128 << 10);
        if (e != cudaSuccess) return cuda_fail(e, "sort shared memory");
        k_onemove_compact_sort<<<(int)std::min<int64_t>((n + wpb - 1) / wpb, 152 * 16), 32 * wpb, sh, st>>>(n, L.cap1, tile, L.cnt_n1,
                                                                                                          L.n1_st, L.n1);
        k_n1_self<<<L.grid, 256, 0, st>>>(n, L.cnt_n1, L.n1, self);
    }
    dev_free(b, L.n1_st);
    L.n1_st = nullptr;
    DevSpecies &D = b.dev.sp[t];
    D.fw_off = L.cnt_fw;
    D.n1_off = L.cnt_n1;
    D.n1 = L.n1;
    D.n1_self = self;
    (void)S;
    return CIH_OK;
}

int lists_phase3(cih_basis &b, int t, SpeciesBuild &S, Lists &L, cudaStream_t st)
{
    const int64_t n = L.n;
    DevSpecies &D = b.dev.sp[t];
    int rc;
    int32_t *tb, *lev;
    int2 *rec;
    if ((rc = dev_alloc(b, &tb, L.tot[0])) || (rc = dev_alloc(b, &rec, L.tot[0])) ||
        (rc = dev_alloc(b, &lev, (size_t)n * D.NL)))
        return rc;
    if (n > 0) {
        count_launches(1);
        with_words(b.W, [&](auto w) {
            k_split<decltype(w)::value><<<L.grid, 256, 0, st>>>(
                S, D.orb_base, D.N0, D.NL, L.d_cls_of, L.d_class_stage, L.cnt_fw, L.fw_st, t == 0 ? b.dev.rowbase : nullptr,
                t == 0 ? b.dev.nb : nullptr, b.dev.pid, b.dev.gsize, b.dev.goff, b.dev.ntot, rec, tb, lev, b.dev_status);
        });
    }
    dev_free(b, L.fw_st);
    L.fw_st = nullptr;
    D.fw_rec = rec;
    D.fw_tb = tb;
    D.fw_lev = lev;
    return CIH_OK;
}

void species_prep(const cih_basis &b, int t, SpeciesHost &H)
{
    const int W = b.W;
    const Species &s = b.s[t];
    H.bits.resize((size_t)s.n_sd * W);               // bit strings compacted to W words
    for (int64_t i = 0; i < s.n_sd; ++i)
        for (int w = 0; w < W; ++w) H.bits[i * W + w] = s.bits[i * kMaxWords + w];
    H.N.assign(s.N.begin(), s.N.end());
    H.M2.assign(s.M2.begin(), s.M2.end());
    H.cls_end.resize(s.n_sd);
    for (int64_t i = 0; i < s.n_sd; ++i) H.cls_end[i] = s.cls_end[s.cls[i]];
    H.cb.assign(s.cls_begin.begin(), s.cls_begin.end());
    H.ce.assign(s.cls_end.begin(), s.cls_end.end());
    H.oN.assign(s.oN.begin(), s.oN.end());
    H.om2.assign(s.om2.begin(), s.om2.end());
    for (int m : s.cls_M2) H.mtop = std::max(H.mtop, std::abs(m));
    H.keep.assign((size_t)(2 * H.mtop + 1) * (s.Nsub_max + 1), 0);
    for (int64_t i = 0; i < s.n_sd; ++i) H.keep[(size_t)(s.M2[i] + H.mtop) * (s.Nsub_max + 1) + s.N[i]] = 1;
    H.cls_of.resize(std::max<int64_t>(s.n_sd, 1));
    H.class_stage.resize(std::max<size_t>(s.cls_begin.size(), 1));
    for (size_t c = 0; c < s.cls_begin.size(); ++c) {
        const int64_t m = s.cls_end[c] - s.cls_begin[c];
        H.class_stage[c] = H.fw_stage;
        H.fw_stage += m * (m - 1) / 2;
        for (int64_t x = s.cls_begin[c]; x < s.cls_end[c]; ++x) H.cls_of[x] = (int32_t)c;
    }
}

int species_upload(cih_basis &b, int t, const SpeciesHost &H, Lists &L, cudaStream_t st)
{
    const int W = b.W;
    const Species &s = b.s[t];
    int rc;
    uint64_t *d_bits; int8_t *d_N; int16_t *d_M2; int32_t *d_cls_end, *d_cb, *d_ce;
    int8_t *d_oN; int16_t *d_om2;
    int32_t *d_upto;
    uint8_t *d_keep;
    int maxN = 0;
    for (int a = 0; a < s.n_orb; ++a) maxN = std::max(maxN, s.oN[a]);
    std::vector<int32_t> upto(maxN + 1, 0);
    for (int a = 0; a < s.n_orb; ++a) upto[s.oN[a]] += 1;
    for (int k = 1; k <= maxN; ++k) upto[k] += upto[k - 1];
    for (int a = 1; a < s.n_orb; ++a)
        if (s.oN[a] < s.oN[a - 1]) return fail(CIH_ERR_UNSUPPORTED, "orbitals not ordered by shell");
    Packer up(b, st);
    up.add(&d_bits, H.bits);
    up.add(&d_N, H.N);
    up.add(&d_M2, H.M2);
    up.add(&d_cls_end, H.cls_end);
    up.add(&d_cb, H.cb);
    up.add(&d_ce, H.ce);
    up.add(&d_oN, H.oN);
    up.add(&d_om2, H.om2);
    up.add(&d_upto, upto);
    up.add(&d_keep, H.keep);
    up.add(&L.d_cls_of, H.cls_of);
    up.add(&L.d_class_stage, H.class_stage);
    if ((rc = up.flush())) return rc;
    DevSpecies &D = b.dev.sp[t];
    D.bits = d_bits;
    D.N = d_N;
    D.cls_end = d_cls_end;
    D.n_sd = (int32_t)s.n_sd;
    D.n_orb = s.n_orb;
    D.orb_base = t == 0 ? 0 : b.s[0].n_orb;
    D.N0 = s.N0;
    D.NL = s.Z > 0 ? ((s.Nsub_max - s.N0) >> 1) + 1 : 1;
    if (D.NL > kLevels) return fail(CIH_ERR_UNSUPPORTED, "internal: more oscillator levels than 256 orbitals give");

    SpeciesBuild S{d_bits, d_N, d_M2, d_cls_end, d_cb, d_ce, d_oN, d_om2, (int32_t)s.n_sd, s.n_orb, s.Nsub_max};
    uint32_t cap = 64;
    while (cap < 2 * (uint64_t)s.n_sd) cap <<= 1;
    int32_t *table;
    if ((rc = dev_alloc(b, &table, cap))) return rc;
    if (cudaMemsetAsync(table, 0xFF, sizeof(int32_t) * cap, st) != cudaSuccess)
        return cuda_fail(cudaGetLastError(), "hash table");
    S.hash = table;
    S.hash_mask = cap - 1;
    uint64_t *fold = nullptr;
    if (W > 1) {
        if ((rc = dev_alloc(b, &fold, s.n_sd))) return rc;
        if (s.n_sd > 0) {
            count_launches(1);
            k_fold<<<(int)std::min<int64_t>((s.n_sd + 255) / 256, 65535), 256, 0, st>>>(s.n_sd, W, d_bits, fold);
        }
    }
    S.fold = fold;
    S.orb_upto = d_upto;
    S.keep = d_keep;
    S.mtop = H.mtop;
    S.maxN = maxN;
    const int hg = (int)std::min<int64_t>((s.n_sd + 255) / 256 + 1, 65535);
    count_launches(1);
    with_words(W, [&](auto w) { k_hash_build<decltype(w)::value><<<hg, 256, 0, st>>>(S, table); });
    b.sbuild[t] = S;
    return CIH_OK;
}

// tables that need the partner ranges, the table layout and the pn split
int basis_tables_upload(cih_basis &b, cudaStream_t st)
{
    int rc;
    int ntot = b.s[0].n_orb + b.s[1].n_orb;
    std::vector<int8_t> orbN(ntot);
    for (int a = 0; a < ntot; ++a) orbN[a] = (int8_t)(a < b.s[0].n_orb ? b.s[0].oN[a] : b.s[1].oN[a - b.s[0].n_orb]);
    int32_t *d_nb, *d_nc, *d_pid, *d_gsize;
    int64_t *d_rowbase, *d_goff;
    int8_t *d_orbN;
    Packer up(b, st);
    up.add(&d_nb, b.nb);
    up.add(&d_nc, b.nc);
    up.add(&d_rowbase, b.rowbase);
    up.add(&d_orbN, orbN);
    up.add(&d_pid, b.layout.pid);
    up.add(&d_gsize, b.layout.gsize);
    up.add(&d_goff, b.layout.goff);
    b.dev.ngroups = (int32_t)b.layout.gsize.size();
    b.dev.n_p = (int32_t)b.s[0].n_sd;
    b.dev.ntot = ntot;
    b.dev.dim = b.dim;
    b.dev.tbme_len = b.layout.total;
    b.dev.Nlim = b.Nlim;
    b.dev.A = b.space.Z + b.space.N;
    b.dev.nZ[0] = b.space.Z;
    b.dev.nZ[1] = b.space.N;
    // pn pairs by proton orbital and neutron type t = (2m, N parity)
    const Species &P = b.s[0], &Q = b.s[1];
    int mtop = 1;                                              // odd, >= every |2m|
    for (int c = 0; c < Q.n_orb; ++c) mtop = std::max(mtop, std::abs(Q.om2[c]));
    const int T = b.dev.pn_T = (mtop + 1) * 2;
    if (T > 32) return fail(CIH_ERR_UNSUPPORTED, "neutron orbitals with 2m above 15");
    std::vector<uint16_t> orbs(std::max(Q.n_orb, 1), 0);       // r(b) | t(b) << 8
    std::vector<int32_t> pcode(std::max(P.n_orb, 1), 0), ncode(std::max(Q.n_orb, 1), 0);
    for (int c = 0; c < Q.n_orb; ++c) {
        const int r = b.pn.rn[c], t = ((Q.om2[c] + mtop) / 2) * 2 + (Q.oN[c] & 1);
        orbs[c] = (uint16_t)(r | t << 8);
        ncode[c] = r | r << 8 | t << 16 | t << 21;
    }
    int ptop = 1;
    for (int a = 0; a < P.n_orb; ++a) ptop = std::max(ptop, std::abs(P.om2[a]));
    if (ptop > 15) return fail(CIH_ERR_UNSUPPORTED, "proton orbitals with 2m above 15");
    std::vector<int2> pk(64, make_int2(0, 0));                 // group of (a, t): key (t + 2 m'_a) ^ N_a parity
    std::vector<int16_t> ps((size_t)std::max(P.n_orb, 1) * T, 0);
    std::vector<uint8_t> pa(std::max(P.n_orb, 1), 0);          // N_a parity | 2 m'_a << 1, m'_a = (2m_a + ptop) / 2
    for (int a = 0; a < P.n_orb; ++a) {
        pa[a] = (uint8_t)((P.oN[a] & 1) | (P.om2[a] + ptop) << 1);
        pcode[a] = a | a << 8 | pa[a] << 17;
        for (int t = 0; t < T; ++t) {
            const int m = 2 * (t >> 1) - mtop, k2 = P.om2[a] + m + b.pn.m2span;
            if (k2 < 0 || k2 > 2 * b.pn.m2span) continue;
            const int kappa = (k2 / 2) * 2 + ((P.oN[a] + t) & 1);
            pk[(t + (pa[a] >> 1)) ^ (pa[a] & 1)] = make_int2(b.pn.goff[kappa], b.pn.gsize[kappa]);
            ps[(size_t)a * T + t] = b.pn.S[(size_t)a * b.pn.G + kappa];
        }
    }
    // the groups as full squares, one after another (the fill's working copy of the pn channel)
    std::vector<int2> pq(64, make_int2(0, 0));
    std::vector<int32_t> sqrow;                                // every row of every square: group << 16 | row
    int64_t sq = 0;
    for (int k = 0; k < 64; ++k) {
        pq[k] = make_int2((int)std::min<int64_t>(sq, INT32_MAX), pk[k].y);
        sq += (int64_t)pk[k].y * pk[k].y;
        for (int u = 0; u < pk[k].y; ++u) sqrow.push_back(k << 16 | u);
    }
    b.sq_total = sq;
    b.dev.n_sqrow = (int32_t)sqrow.size();
    int2 *d_pk, *d_pq; int16_t *d_ps; uint16_t *d_orbs; uint8_t *d_pa; int32_t *d_sqrow, *d_pc, *d_nc2;
    int16_t *d_obg, *d_obl; int32_t *d_obs, *d_obo;
    up.add(&d_pq, pq);
    up.add(&d_sqrow, sqrow);
    up.add(&d_pc, pcode);
    up.add(&d_nc2, ncode);
    up.add(&d_pk, pk);
    up.add(&d_ps, ps);
    up.add(&d_orbs, orbs);
    up.add(&d_pa, pa);
    up.add(&d_obg, b.onebody.grp);
    up.add(&d_obl, b.onebody.loc);
    up.add(&d_obs, b.onebody.gsize);
    up.add(&d_obo, b.onebody.goff);
    if ((rc = up.flush())) return rc;
    b.dev.nb = d_nb;
    b.dev.nc = d_nc;
    b.dev.rowbase = d_rowbase;
    b.dev.orbN = d_orbN;
    b.dev.pid = d_pid;
    b.dev.gsize = d_gsize;
    b.dev.goff = d_goff;
    b.dev.pn_kq = d_pq;
    b.dev.sqrow = d_sqrow;
    b.dev.code[0] = d_pc;
    b.dev.code[1] = d_nc2;
    b.dev.pn_k = d_pk;
    b.dev.pn_a = d_pa;
    b.dev.pn_s = d_ps;
    b.dev.orbs = d_orbs;
    b.dev.ob_grp = d_obg;
    b.dev.ob_loc = d_obl;
    b.dev.ob_gsize = d_obs;
    b.dev.ob_goff = d_obo;
    return CIH_OK;
}

// Page-locked 8-word slots for the totals read back during set-up, kept for the
// next basis (allocating and freeing pinned memory costs more than the set-up's
// own synchronisations).
std::mutex g_slot_mu;
std::vector<int64_t *> g_slots;

struct PinnedTotals {
    int64_t *p = nullptr;
    cudaStream_t st = nullptr;                // copies into the slot are queued here
    cudaError_t get()
    {
        {
            std::lock_guard<std::mutex> lock(g_slot_mu);
            if (!g_slots.empty()) {
                p = g_slots.back();
                g_slots.pop_back();
                return cudaSuccess;
            }
        }
        cudaError_t e = cudaHostAlloc((void **)&p, 8 * sizeof(int64_t), cudaHostAllocPortable);   // any device
        if (e != cudaSuccess) p = nullptr;
        return e;
    }
    ~PinnedTotals()
    {
        if (!p) return;
        cudaStreamSynchronize(st);            // no copy still in flight into a returned slot
        std::lock_guard<std::mutex> lock(g_slot_mu);
        g_slots.push_back(p);
    }
};

// A second stream for the neutron species' list passes, which need nothing of the
// proton species'.  The destructor waits for
// it, so that no early return leaves its kernels running on buffers the basis
// then frees.
struct SideStream {
    cudaStream_t s = nullptr;
    cudaEvent_t ev[3] = {nullptr, nullptr, nullptr};
    cudaError_t create()
    {
        cudaError_t e = cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking);
        if (e != cudaSuccess) { s = nullptr; return e; }
        for (auto &x : ev)
            if ((e = cudaEventCreateWithFlags(&x, cudaEventDisableTiming)) != cudaSuccess) { x = nullptr; return e; }
        return cudaSuccess;
    }
    ~SideStream()
    {
        if (s) cudaStreamSynchronize(s);
        for (auto x : ev)
            if (x) cudaEventDestroy(x);
        if (s) cudaStreamDestroy(s);
    }
};

// device allocations and frees of a block of calls go to stream s
struct AllocOn {
    cih_basis &b;
    cudaStream_t old;
    AllocOn(cih_basis &b_, cudaStream_t s) : b(b_), old(b_.stream) { b.stream = s; }
    ~AllocOn() { b.stream = old; }
};

}  // namespace

int upload_and_build_neighbours(cih_basis &b, cudaStream_t st, const std::function<int()> &host_rest)
{
    int rc;
    const int W = b.W;
    b.stream = st;
    if ((rc = device_pool(b.device, &b.pool))) return rc;
    Timer tm("basis device set-up");
    if ((rc = dev_alloc(b, &b.dev_status, 4))) return rc;
    if (cudaMemsetAsync(b.dev_status, 0, 4 * sizeof(int), st) != cudaSuccess) return cuda_fail(cudaGetLastError(), "status");
    PinnedTotals pin;
    pin.st = st;
    cudaError_t e = pin.get();
    if (e != cudaSuccess) return cuda_fail(e, "pinned totals");
    for (int i = 0; i < 8; ++i) pin.p[i] = 0;
    Lists L[2];
    L[0].tot = pin.p;
    L[1].tot = pin.p + 3;
    // every kernel reads W words per bit string: they must hold every orbital
    for (int t = 0; t < 2; ++t)
        if (64 * W < b.s[t].n_orb || (W != 1 && W != 2 && W != 4))
            return fail(CIH_ERR_UNSUPPORTED, "internal: bit strings of " + std::to_string(W) + " words for " +
                                                 std::to_string(b.s[t].n_orb) + " orbitals");
    // 1. per species, protons on st and neutrons on a second stream: upload,
    //    hash table, staged passes (queued, no synchronisation).  Uploads from
    //    pageable memory wait for their own stream only, so neither species'
    //    uploads wait for the other's kernels.
    SpeciesHost H[2];
    side_by_side([&]() { species_prep(b, 0, H[0]); }, [&]() { species_prep(b, 1, H[1]); }, small_host(b.s[0].n_sd + b.s[1].n_sd));
    SideStream side;
    if ((e = side.create()) != cudaSuccess) return cuda_fail(e, "side stream");
    const cudaStream_t ss[2] = {st, side.s};
    cudaEventRecord(side.ev[0], st);                   // after the status words are cleared
    cudaStreamWaitEvent(side.s, side.ev[0], 0);
    tm.mark("species host arrays");
    for (int t = 0; t < 2; ++t) {
        AllocOn on(b, ss[t]);
        if ((rc = species_upload(b, t, H[t], L[t], ss[t]))) return rc;
        with_words(W, [&](auto w) { rc = lists_phase1<decltype(w)::value>(b, t, b.sbuild[t], H[t], L[t], ss[t]); });
        if (rc) return rc;
    }
    tm.mark("species queued");
    // host work that the kernels above do not need: ranges, table layout, pn split
    if ((rc = host_rest())) return rc;
    tm.mark("host ranges + layout");
    e = cudaStreamSynchronize(st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(side.s);
    if (e != cudaSuccess) return cuda_fail(e, "neighbour counts");
    tm.mark("staged passes done");
    // basis tables while both streams are idle (no upload waits for a kernel)
    if ((rc = basis_tables_upload(b, st))) return rc;
    cudaEventRecord(side.ev[1], st);
    {
        const Species &Q = b.s[1];
        int dm = 0;
        for (int x = 0; x < Q.n_orb; ++x)
            for (int y = 0; y < Q.n_orb; ++y) dm = std::max(dm, std::abs(Q.om2[x] - Q.om2[y]));
        b.dev.DM = dm;
        b.dev.dir_len = 1 + (dm + 1) * 2 * b.dev.sp[1].NL;
        if (b.dev.dir_len > 65535) return fail(CIH_ERR_UNSUPPORTED, "neutron bucket directory too long");
    }
    // 2. exact-size lists, 3. forward lists split, with two-move indices (these
    //    read the basis tables), again one species per stream
    for (int t = 0; t < 2; ++t) {
        AllocOn on(b, ss[t]);
        if ((rc = lists_phase2(b, t, b.sbuild[t], L[t], ss[t]))) return rc;
        if (t == 1) cudaStreamWaitEvent(side.s, side.ev[1], 0);
        if ((rc = lists_phase3(b, t, b.sbuild[t], L[t], ss[t]))) return rc;
    }
    b.scan_scratch_len = scan_scratch_needed(b.dim);
    if ((rc = dev_alloc(b, &b.scan_scratch, b.scan_scratch_len))) return rc;
    {
        // neutrons: packed one-move lists, their bucket directory, records and
        // occupied lists, on the second stream
        const int64_t nn = b.s[1].n_sd, tot = L[1].tot[1];
        int2 *n1p;
        int16_t *dir;
        uint8_t *occn;
        int32_t *occc;
        NeutronRec *nrec;
        const int g1 = (int)std::min<int64_t>((nn + 255) / 256 + 1, 65535);
        AllocOn on(b, side.s);
        if ((rc = dev_alloc(b, &n1p, tot)) || (rc = dev_alloc(b, &dir, (size_t)nn * b.dev.dir_len)) ||
            (rc = dev_alloc(b, &nrec, nn)) || (rc = dev_alloc(b, &occn, (size_t)nn * std::max(b.s[1].Z, 1))) ||
            (rc = dev_alloc(b, &occc, (size_t)nn * std::max(b.s[1].Z, 1))))
            return rc;
        if (nn > 0) {
            const DevSpecies &D = b.dev.sp[1];
            const SpeciesBuild &SB = b.sbuild[1];
            count_launches(4);
            with_words(W, [&](auto w) {
                k_n1_pack<decltype(w)::value><<<grid_for(nn), 256, 0, side.s>>>(SB, D.n1_off, D.n1, b.dev.orbs, n1p);
                k_occ<decltype(w)::value><<<g1, 256, 0, side.s>>>(SB, b.s[1].Z, b.dev.code[1], occn, occc);
            });
            k_dir<<<grid_for(nn), 256, 0, side.s>>>(SB, D.n1_off, D.n1, D.N0, D.NL, b.dev.DM, b.dev.dir_len, dir);
            k_neutron_rec<<<g1, 256, 0, side.s>>>(D, nrec);
        }
        b.dev.occ[1] = occn;
        b.dev.occ_code[1] = occc;
        b.dev.n1p = n1p;
        b.dev.dir = dir;
        b.dev.nrec = nrec;
        cudaEventRecord(side.ev[2], side.s);           // the neutron half is complete here
    }
    tm.mark("neutron lists queued");
    {
        // protons (which read no neutron list): occupied lists, rows, groups, records
        const int64_t np = b.s[0].n_sd;
        const int g0 = (int)std::min<int64_t>((np + 255) / 256 + 1, 65535);
        int64_t *goff;
        int32_t *row_p;
        int2 *walk = nullptr;
        uint8_t *occp;
        int32_t *occc;
        int2 *l1;
        ProtonRec *prec;
        if ((rc = dev_alloc(b, &goff, np + 1)) || (rc = dev_alloc(b, &row_p, b.dim)) ||
            (rc = dev_alloc(b, &occp, (size_t)np * std::max(b.s[0].Z, 1))) ||
            (rc = dev_alloc(b, &occc, (size_t)np * std::max(b.s[0].Z, 1))) || (rc = dev_alloc(b, &l1, L[0].tot[1])) ||
            (rc = dev_alloc(b, &prec, np)) || (b.dim >= kWalkRows && (rc = dev_alloc(b, &walk, b.dim))))
            return rc;
        const int grid = grid_for(np);
        const SpeciesBuild &SB = b.sbuild[0];
        if (np > 0) {
            count_launches(3);
            with_words(W, [&](auto w) {
                k_groups<decltype(w)::value, 0><<<grid, 256, 0, st>>>(SB, b.dev, goff, nullptr, nullptr);
                k_occ<decltype(w)::value><<<g0, 256, 0, st>>>(SB, b.s[0].Z, b.dev.code[0], occp, occc);
            });
            k_row_p<<<grid, 256, 0, st>>>(np, b.dev.rowbase, b.dev.nb, b.dev.nc, row_p, walk);
        }
        if ((rc = exclusive_scan_i64(goff, np, b.scan_scratch, b.scan_scratch_len, st))) return rc;
        int64_t *total = pin.p + 6;
        e = cudaMemcpyAsync(total, goff + np, sizeof(int64_t), cudaMemcpyDeviceToHost, st);
        if (e == cudaSuccess) e = cudaStreamSynchronize(st);
        if (e != cudaSuccess) return cuda_fail(e, "group count");
        int4 *grp;
        if ((rc = dev_alloc(b, &grp, *total))) return rc;
        if (np > 0) {
            count_launches(2);
            with_words(W, [&](auto w) {
                k_groups<decltype(w)::value, 1><<<grid, 256, 0, st>>>(SB, b.dev, goff, grp, l1);
            });
            k_proton_rec<<<g0, 256, 0, st>>>(b.dev, goff, prec);
        }
        tm.mark("groups queued");
        b.dev.occ[0] = occp;
        b.dev.occ_code[0] = occc;
        for (int t = 0; t < 2; ++t) {
            b.fw_total[t] = L[t].tot[0];
            b.n1_total[t] = L[t].tot[1];
        }
        b.dev.row_p = row_p;
        b.dev.walk = walk;
        b.dev.grp = grp;
        b.dev.l1 = l1;
        b.dev.prec = prec;
    }
    cudaStreamWaitEvent(st, side.ev[2], 0);            // join: later work on st sees both species
    e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return cuda_fail(e, "basis upload");
    return CIH_OK;
}

}  // namespace cih
