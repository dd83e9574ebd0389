// normal64.cuh -- binary64 Box-Muller normals from integer arithmetic.
//
// GB300's binary64 pipe takes 64 cycles of a sub-partition per warp
// instruction (two lanes per clock and SM); log, sqrt and sincospi of one pair
// of normals occupied it for about 70 of the 80 binary64 operations of an
// Euler-Maruyama step.  Here the pair is computed on the integer units in
// 64-bit fixed point and only then turned into binary64, so that the pipe is
// left to the step itself:
//   radius  r(u0) = sqrt(-2 ln u0), 2^-60 units: a polynomial of degree 7 per
//           segment (46 binades of u0 and 1 - u0 x 32), Horner with a 31-bit
//           argument;
//   angle   2 pi u1 = quarter turns + node + b: cos and sin of the 1024 nodes
//           of a quarter turn in 2^-63 units, of b < 2^-9 from its series, and
//           the addition formulas.
// The normals are within 2^-57 of the exact ones (2^-58.5 rms), below the
// rounding of a binary64 number of their size except where |z| < 2^-4.
// Tables and constants: normal_tables.py (the header it writes is included by
// the translation unit that holds the tables).
#pragma once

#include <stdint.h>

#ifdef __CUDA_ARCH__
#define PR_CLZ(v) __clz((int)(v))
#define PR_UMULHI(a, b) __umulhi((a), (b))
#define PR_SMULHI(a, b) __mulhi((a), (b))
#else
#define PR_CLZ(v) __builtin_clz(v)
#define PR_UMULHI(a, b) ((uint32_t)(((uint64_t)(a) * (uint64_t)(b)) >> 32))
#define PR_SMULHI(a, b) ((int32_t)(((int64_t)(a) * (int64_t)(b)) >> 32))
#endif

#ifdef __CUDACC__
#define PR_HD __host__ __device__ __forceinline__
#else
#define PR_HD inline
#endif

namespace pr {

constexpr int kNormalTableWords = 6 * kRadiusSegments + 2 * kNodes + kRadiusSegments / 2;

struct alignas(16) U64x2 {
    uint64_t a, b;
};

// The tables, 16-byte aligned, in the order the header holds them.
struct NormalTables {
    const U64x2* radius;   // [kRadiusSegments][3]
    const U64x2* nodes;    // [kNodes] (cos, sin)
    const int32_t* c7;     // [kRadiusSegments]
};

PR_HD NormalTables normal_tables_at(const void* base)
{
    NormalTables t;
    t.radius = static_cast<const U64x2*>(base);
    t.nodes = t.radius + 3 * kRadiusSegments;
    t.c7 = reinterpret_cast<const int32_t*>(t.nodes + kNodes);
    return t;
}

// floor(acc t / 2^32) + c for a signed acc and 0 <= t < 2^31
PR_HD int64_t horner_step(int64_t acc, uint32_t t, uint64_t c)
{
    const int64_t hi = (int64_t)(int32_t)(acc >> 32) * (int64_t)(int32_t)t;
    return hi + (int64_t)(c + PR_UMULHI((uint32_t)acc, t));
}

// a b / 2^64 for a < 2^63 + 1, b < 2^63, to within two units below
PR_HD uint64_t mulhi_near(uint64_t a, uint64_t b)
{
    const uint32_t al = (uint32_t)a, ah = (uint32_t)(a >> 32), bl = (uint32_t)b, bh = (uint32_t)(b >> 32);
    const uint64_t mid = (uint64_t)ah * bl + (uint64_t)al * bh;
    return (uint64_t)ah * bh + (mid >> 32);
}

// r 2^60 for the uniform (2 (w >> 9) + 1) 2^-24
PR_HD uint64_t radius_fixed(uint32_t w, const NormalTables& tab)
{
    const uint32_t m = (w >> 8) | 1u;
    const uint32_t side = w >> 31;
    const uint32_t v = side ? (1u << 24) - m : m;
    const int lz = PR_CLZ(v);
    const uint32_t norm = v << lz;                     // leading bit at 31
    const uint32_t t = (norm << (kSegBits + 1)) >> 1;
    const int g = (int)(((side ? 23u : 0u) + (uint32_t)(31 - lz)) << kSegBits) +
                  (int)((norm >> (31 - kSegBits)) & ((1u << kSegBits) - 1u));
    const U64x2 c01 = tab.radius[3 * g], c23 = tab.radius[3 * g + 1], c4t = tab.radius[3 * g + 2];
    int32_t q = tab.c7[g];
    q = (int32_t)(c4t.b >> 32) + PR_SMULHI(q, (int32_t)t);
    q = (int32_t)(uint32_t)c4t.b + PR_SMULHI(q, (int32_t)t);
    int64_t acc = (int64_t)c4t.a + (((int64_t)q * (int64_t)(int32_t)t) >> (32 - kTailShift));
    acc = horner_step(acc, t, c23.b);
    acc = horner_step(acc, t, c23.a);
    acc = horner_step(acc, t, c01.b);
    return (uint64_t)horner_step(acc, t, c01.a);
}

// |cos| 2^63, |sin| 2^63 of 2 pi u and the quarter turn, u = (2 (w >> 9) + 1) 2^-24:
// cos(2 pi u) = (+c, -s, -c, +s)[quarter], sin(2 pi u) = (+s, +c, -s, -c)[quarter]
PR_HD uint32_t angle_fixed(uint32_t w, const NormalTables& tab, uint64_t& c, uint64_t& s)
{
    const U64x2 node = tab.nodes[(w >> 20) & 1023u];
    const uint32_t n = ((w >> 8) & 4095u) | 1u;        // b = n 2 pi 2^-24
    const uint32_t n2 = n * n, n2s = n2 << 8;
    const uint32_t k3 = (uint32_t)kSin3 - (PR_UMULHI(n2s, (uint32_t)kSin5) >> 16);
    const uint64_t k1 = kSin1 - PR_UMULHI(n2s, k3);    // sin(b) / n, 2^-73 units
    const uint64_t sb = (((uint64_t)((uint32_t)(k1 >> 32) * n) << 32) + (uint64_t)(uint32_t)k1 * n) >> 9;
    const uint64_t k2 = kCos2 - PR_UMULHI(n2s, (uint32_t)kCos4);   // (1 - cos b) / n^2, 2^-97 units
    const uint64_t e = ((uint64_t)(uint32_t)(k2 >> 32) * n2 + PR_UMULHI((uint32_t)k2, n2)) >> 1;
    c = node.a - mulhi_near(node.a, e) - mulhi_near(node.b, sb);
    s = node.b - mulhi_near(node.b, e) + mulhi_near(node.a, sb);
    return w >> 30;
}

// The encoding of v 2^-59 (v > 0) rounded to nearest, ties up; `sign` in bit 31
PR_HD uint64_t encode_2m59(uint64_t v, uint32_t sign)
{
    uint32_t hi = (uint32_t)(v >> 32);
    int lz = 0;
    if (hi == 0u) {   // below 2^-27: rare
        v <<= 32;
        hi = (uint32_t)(v >> 32);
        lz = 32;
    }
    const int z = PR_CLZ(hi | 1u);
    v <<= z;
    const uint64_t bits = (v >> 11) + ((v >> 10) & 1u);
    return bits + ((uint64_t)(((uint32_t)(1026 - lz - z) << 20) | sign) << 32);
}

// The normals z0 = r cos, z1 = r sin of the words w0 (radius) and w1 (angle).
PR_HD void box_muller_fixed(uint32_t w0, uint32_t w1, const NormalTables& tab, uint64_t& z0, uint64_t& z1)
{
    const uint64_t r = radius_fixed(w0, tab);
    uint64_t c, s;
    const uint32_t q = angle_fixed(w1, tab, c, s);
    const uint64_t a = mulhi_near(r, q & 1u ? s : c), b = mulhi_near(r, q & 1u ? c : s);
    z0 = encode_2m59(a, ((q + 1u) & 2u) << 30);
    z1 = encode_2m59(b, (q & 2u) << 30);
}

}  // namespace pr
