// normal64.cuh -- binary64 Box-Muller normals from integer arithmetic.
//
// GB300's binary64 pipe takes 64 cycles of a sub-partition per warp
// instruction (two lanes per clock and SM); log, sqrt and sincospi of one pair
// of normals occupied it for about 70 of the 80 binary64 operations of an
// Euler-Maruyama step.  Here the pair is computed on the integer units in
// 64-bit fixed point and only then turned into binary64, so that the pipe is
// left to the step itself:
//   radius  r(u0) = sqrt(-2 ln u0): a polynomial of degree 7 per segment (46
//           binades of u0 and 1 - u0 x 32), Horner with a 31-bit argument, in
//           units of 2^-(60 + shift) that leave r 61 bits at least in every
//           binade;
//   angle   2 pi u1 reflected into an eighth of a turn = node + b: cos and sin of
//           the 1024 nodes, of b < 2^-10.3 from its series, and the addition
//           formulas.  The sine is a sum of positive terms there; its terms are
//           scaled by 2^z, z the leading zeros of the angle, so that it keeps
//           its bits where it is small.
// So the normals have the same relative error at every size: before the one
// rounding to binary64 2^-58.6 rms and 2^-55.3 at most, after it 2^-54.2 rms (in
// absolute fixed point a small normal loses bits: 2^-47.5 rms, 2^-41 below 2^-12).
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
    const U64x2* nodes;    // [kNodes] (cos 2^63, sin 2^(62 + z))
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

// a b / 2^64 for a < 2^63, b <= 2^63, to within two units below
PR_HD uint64_t mulhi_near(uint64_t a, uint64_t b)
{
    const uint32_t al = (uint32_t)a, ah = (uint32_t)(a >> 32), bl = (uint32_t)b, bh = (uint32_t)(b >> 32);
    const uint64_t mid = (uint64_t)ah * bl + (uint64_t)al * bh;
    return (uint64_t)ah * bh + (mid >> 32);
}

// r 2^(60 + shift) for the uniform (2 (w >> 9) + 1) 2^-24
PR_HD uint64_t radius_fixed(uint32_t w, const NormalTables& tab, uint32_t& shift)
{
    const uint32_t m = (w >> 8) | 1u;
    const uint32_t side = w >> 31;
    const uint32_t v = side ? (1u << 24) - m : m;
    const int lz = PR_CLZ(v);
    shift = side ? (uint32_t)(lz - 5) >> 1 : (lz < 19 ? 1u : 0u);   // radius_shift(side, 31 - lz)
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

// cos 2^63 and sin 2^(62 + z) of the angle 2 pi u reflected into the first eighth
// of a turn, u = (2 (w >> 9) + 1) 2^-24; z such that the sine is between 2^60.4 and
// 2^61.7
PR_HD void angle_fixed(uint32_t w, const NormalTables& tab, uint64_t& c, uint64_t& s, uint32_t& z)
{
    const uint32_t x = (w >> 8) ^ (uint32_t)((int32_t)(w << 2) >> 31);   // odd eighths run backwards
    const U64x2 node = tab.nodes[(x >> 11) & 1023u];
    const uint32_t n = (x & 2047u) | 1u;               // b = n d, d = 2 pi 2^-24
    z = (uint32_t)PR_CLZ((int)((x << 11) | 2048u));    // (the sine is 0.90 to 1 times its angle)
    const uint32_t n2 = n * n, n2s = n2 << 10;
    const uint32_t k3 = (uint32_t)kSin3 - ((PR_UMULHI(n2s, (uint32_t)kSin5) + (1u << 23)) >> 24);
    const uint64_t k1 = kSin1 - (((uint64_t)n2s * k3) >> 24);   // sin(b) / n, 2^-84 units
    const uint64_t k2 = kCos2 - PR_UMULHI(n2s, (uint32_t)kCos4);   // (1 - cos b) / n^2, 2^-97 units
    const uint64_t e = ((uint64_t)(uint32_t)(k2 >> 32) * n2 + PR_UMULHI((uint32_t)k2, n2)) >> 1;   // 1 - cos b, 2^-64
    const uint32_t nz = n << (z + 11u);                // (n below 2^11, and 2^(21 - z) at node 0)
    const uint64_t sb = (uint64_t)(uint32_t)(k1 >> 32) * nz + PR_UMULHI((uint32_t)k1, nz);   // sin b, 2^-(63 + z)
    c = node.a - mulhi_near(node.a, e) - ((mulhi_near(node.b, sb) >> (2u * z)) << 2);
    s = node.b - mulhi_near(node.b, e) + mulhi_near(node.a, sb);
}

// The encoding of v 2^-(59 + shift) rounded to nearest, ties up (2^32 <= v < 2^63)
PR_HD uint64_t encode_2m59(uint64_t v, uint32_t shift)
{
    const int z = PR_CLZ((int)(uint32_t)(v >> 32));
    v <<= z;
    const uint64_t bits = (v >> 11) + ((v >> 10) & 1u);
    return bits + ((uint64_t)((1026u - shift - (uint32_t)z) << 20) << 32);
}

// The normals z0 = r cos, z1 = r sin of the words w0 (radius) and w1 (angle):
// the reflected pair changes places in the odd eighths of a turn, the signs
// are those of the quarter.
PR_HD void box_muller_fixed(uint32_t w0, uint32_t w1, const NormalTables& tab, uint64_t& z0, uint64_t& z1)
{
    uint32_t shift, z;
    const uint64_t r = radius_fixed(w0, tab, shift);
    uint64_t c, s;
    angle_fixed(w1, tab, c, s, z);
    const uint64_t a = encode_2m59(mulhi_near(r, c), shift), b = encode_2m59(mulhi_near(r, s), shift + z - 1u);
    const uint32_t q = w1 >> 30;
    const bool swap = ((w1 >> 30) ^ (w1 >> 29)) & 1u;
    z0 = (swap ? b : a) | ((uint64_t)(((q + 1u) & 2u) << 30) << 32);
    z1 = (swap ? a : b) | ((uint64_t)((q & 2u) << 30) << 32);
}

}  // namespace pr
