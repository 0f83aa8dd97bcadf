// Device helpers of the row kernels (ham.cu): two-body table lookups and the
// double-float value sums.  Not part of the ABI.
#pragma once

#include <cstdint>

#include "cih_internal.h"

namespace cih {

// Table layout caps of the shared-memory copies the kernels keep.
constexpr int kLayoutCap = 512;   // global table groups
constexpr int kOrbCap = 512;      // combined orbitals (two species of at most 256)

// Table index of V(ab, cd) for combined orbitals in any order; false if the
// pairs are not one table entry (a bug in the walk: flagged by the caller).
// The group sizes and offsets come from shared memory (lg: size and offset
// per group, int2) when given and the layout has at most kLayoutCap groups.
__device__ __forceinline__ bool tbme_at(const DevBasis &B, const int2 *lg, int a, int b, int c, int d, int64_t &idx,
                                        int &sign)
{
    if ((unsigned)a >= (unsigned)B.ntot || (unsigned)b >= (unsigned)B.ntot ||
        (unsigned)c >= (unsigned)B.ntot || (unsigned)d >= (unsigned)B.ntot)
        return false;
    int32_t e1 = B.pid[a * B.ntot + b], e2 = B.pid[c * B.ntot + d];
    if (e1 < 0 || e2 < 0) return false;
    int g = (e1 >> 16) & 0xFFF;
    if (g != ((e2 >> 16) & 0xFFF)) return false;
    sign = (((e1 ^ e2) >> 30) & 1) ? -1 : 1;
    int u = e1 & 0xFFFF, v = e2 & 0xFFFF;
    if (u > v) { const int t = u; u = v; v = t; }
    int64_t n, off;
    if (lg && B.ngroups <= kLayoutCap) {
        const int2 q = lg[g];
        n = q.x;
        off = q.y;
    } else {
        n = B.gsize[g];
        off = B.goff[g];
    }
    idx = off + (int64_t)u * n - (int64_t)u * (u - 1) / 2 + (v - u);
    return true;
}

// A sum of FP32 terms carried as the unevaluated pair hi + lo of floats
// (Dekker's two-sum), about 48 significant bits: exact for the value sums here
// (at most a few dozen FP32 terms within 24 binary orders of magnitude), and
// single-precision arithmetic runs at full rate where the GPU's FP64 units are
// few.  The value stored is hi + lo rounded once to FP32.
struct DF {
    float hi, lo;
};
__device__ __forceinline__ DF df_add(DF a, DF b)
{
    const float s = a.hi + b.hi;
    const float bb = s - a.hi;
    const float e = (a.hi - (s - bb)) + (b.hi - bb);
    const float lo = (e + a.lo) + b.lo;
    const float hi = s + lo;
    return DF{hi, lo - (hi - s)};
}
__device__ __forceinline__ DF df_of(float x) { return DF{x, 0.f}; }
__device__ __forceinline__ float df_round(DF v) { return v.hi + v.lo; }

// table index of a pn element from the proton move (l1: a | c << 8 | sign << 16
// | pn_a[a] << 17) and the neutron move (n1: r(d) | r(b) << 8 | t(b) << 16 |
// t(d) << 21 | sign << 26): u(a, b) = S(a, t(b)) + r(b), v(c, d) = S(c, t(d)) +
// r(d) in the group of (a, t(b)); sign = proton move sign ^ neutron move sign.
// KG, S: pn_k, pn_s in shared memory.
__device__ __forceinline__ int pn_index_at(const int2 *KG, const int16_t *S, int T, int l1, int n1, int &sign)
{
    const int t = (n1 >> 16) & 0x1F;
    const int2 g = KG[(t + ((unsigned)l1 >> 18)) ^ ((l1 >> 17) & 1)];
    int u = S[(l1 & 0xFF) * T + t] + ((n1 >> 8) & 0xFF);
    int v = S[((l1 >> 8) & 0xFF) * T + ((n1 >> 21) & 0x1F)] + (n1 & 0xFF);
    if (u > v) { const int s = u; u = v; v = s; }
    sign = ((l1 >> 16) ^ (n1 >> 26)) & 1;
    return g.x + u * g.y - ((u * (u - 1)) >> 1) + (v - u);
}

// the same element in the pn groups stored as full squares (KQ: pn_kq)
__device__ __forceinline__ int pn_square_at(const int2 *KQ, const int16_t *S, int T, int l1, int n1)
{
    const int t = (n1 >> 16) & 0x1F;
    const int2 g = KQ[(t + ((unsigned)l1 >> 18)) ^ ((l1 >> 17) & 1)];
    const int u = S[(l1 & 0xFF) * T + t] + ((n1 >> 8) & 0xFF);
    return g.x + u * g.y + S[((l1 >> 8) & 0xFF) * T + ((n1 >> 21) & 0x1F)] + (n1 & 0xFF);
}

}  // namespace cih
