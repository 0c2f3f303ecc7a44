// Float64 pair terms with their geometry in 64-bit integers.  The float64 pipe issues one warp instruction
// per scheduler in 64 cycles and bounds the float64 pair kernels, while the integer pipes beside it are idle.
// Coordinates are integers in units of 2^-k, 2^(62-k) being a power of two above every coordinate difference
// of the system (fixed_scale): differences are exact, the squared distance keeps 58 to 62 bits, and 1/r, q/r^3
// and the difference itself become float64 by one rounding each.  Float64 operations are left to the sums.
//
// A coordinate is rounded to 2^-(k+1), at most 2^-63 of the range, where float64 rounds it to 2^-54 of
// itself; so a pair nearer than 2^-9 of the range in every coordinate (and coincident charges) is left to
// the float64 form, whose differences are exact there.
#pragma once

#include "rsqrt64.cuh"

namespace psum {

constexpr int kNoFixed = -100000;             // no integer form: every pair takes the float64 form
constexpr uint32_t kFixedNear = 1u << 21;     // high words below: nearer than 2^-9 of the range
constexpr uint32_t kFixedFar = 1u << 30;      // ... from here on: outside the range

// Out of every range: its difference from any coordinate of the range is 2^62 or more, modulo 2^64 too.
constexpr long long kFixedOut = -0x7fffffffffffffffll - 1;

// x 2^k, rounded; kFixedOut from 2^62 on, for infinities and NaN
__host__ __device__ __forceinline__ long long to_fixed(double x, int k) {
    const long long b = f64_bits(x);
    const int e = (int)(b >> 52) & 0x7ff, s = e - 1075 + k;
    const long long m = e ? (b & 0xfffffffffffffll) | (1ll << 52) : 0;
    if (s > 9) return kFixedOut;
    const long long v = s >= 0 ? m << s : s > -54 ? (m + (1ll << (-s - 1))) >> -s : 0;
    return b < 0 ? -v : v;
}

// A coordinate difference as magnitude and sign mask (the magnitude of a negative one is a unit short,
// 2^-53 of the pair's distance at the most), its float64 value on request.
struct FixedDelta {
    uint64_t a;
    uint32_t sign;
};
__host__ __device__ __forceinline__ FixedDelta fixed_delta(long long s, long long t) {
    const long long d = (long long)((uint64_t)s - (uint64_t)t), g = d >> 63;
    FixedDelta r;
    r.a = (uint64_t)(d ^ g);
    r.sign = (uint32_t)(g >> 32) & 0x80000000u;
    return r;
}
__host__ __device__ __forceinline__ int lead_zeros64(uint64_t v) {
    const uint32_t h = (uint32_t)(v >> 32);
    return h ? lead_zeros32(h) : 32 + lead_zeros32((uint32_t)v);
}
// (0 comes out as a quarter of a unit)
__host__ __device__ __forceinline__ double fixed_value(FixedDelta d, int k) {
    const int z = lead_zeros64(d.a);                                   // 2..64
    const uint64_t mant = ((d.a << (z - 1)) + 0x200u) >> 10;           // its leading one in bit 52
    return f64_from((long long)(mant + ((uint64_t)(uint32_t)(1085 - z - k) << 52) + ((uint64_t)d.sign << 32)));
}

// The squared distance R 2^(64 - 2 s) units^2, R in [2^58, 2^62), of differences below 2^62 of which the
// largest is at least kFixedNear 2^32: each is shifted until that one's leading bit is bit 61, and loses the
// square of its low word, 3 units of R together.  (Outside these bounds every function here gives some value
// without meaning: the kernels compute it and throw it away.)
struct FixedR2 {
    uint64_t R;
    int s;
};
__host__ __device__ __forceinline__ FixedR2 fixed_r2(FixedDelta x, FixedDelta y, FixedDelta z, uint32_t high) {
    FixedR2 r;
    const int s = lead_zeros32(high | kFixedNear) - 2;
    r.s = s > 0 ? s : 0;
    const uint64_t a = x.a << r.s, b = y.a << r.s, c = z.a << r.s;
    const uint32_t ah = (uint32_t)(a >> 32), bh = (uint32_t)(b >> 32), ch = (uint32_t)(c >> 32);
    const uint64_t cross = (uint64_t)ah * (uint32_t)a + (uint64_t)bh * (uint32_t)b + (uint64_t)ch * (uint32_t)c;
    r.R = (uint64_t)ah * ah + (uint64_t)bh * bh + (uint64_t)ch * ch + (cross >> 31);
    return r;
}
// The float32 copy of R 2^-32 for the estimate of its inverse square root.
__host__ __device__ __forceinline__ float fixed_estimate_arg(uint64_t R) {
    const uint32_t h = (uint32_t)(R >> 32);
    return (float)(h > 1u << 26 ? h : 1u << 26);
}

// mantissa M (leading one in bit 63 - z) times 2^(x - 1) with bit 52 as the unit, rounded
__host__ __device__ __forceinline__ double fixed_assemble(uint64_t M, int z, int x) {
    const uint64_t mant = ((M >> (10 - z)) + 1) >> 1;
    return f64_from((long long)(mant + ((uint64_t)(uint32_t)x << 52)));
}

// 1/r and 1/r^3 from the bits yb of a float32 estimate y of (R 2^-32)^(-1/2), relative error below 2^-21:
// with e = 1 - R 2^-32 y^2 (its integer is minus the product's low 64 bits, the leading one cancelling),
//   (R 2^-32)^(-1/2) = y (1 + e/2 + (3/8) e^2) + O((5/16) e^3), the rest below 2^-64;
// the cube from its 62-bit mantissa, and a charge's product with it, in integers too.  Errors before the
// rounding to 53 bits: 2^-57 for 1/r, 2^-55 for q/r^3.
struct FixedInverse {
    uint64_t M;      // 1/r = M 2^(E - 237 + s + k), M in [2^62 - 2^41, 2^63 + 2^42]
    int x;           // E + s + k
    int E;
};
__host__ __device__ __forceinline__ FixedInverse fixed_inverse(FixedR2 r, int k, uint32_t yb) {
    FixedInverse v;
    v.E = (int)(yb >> 23);                                             // y = m 2^(E - 150), E in 111..114
    const uint32_t m = (yb & 0x7fffffu) | 0x800000u;
    const uint64_t mm = (uint64_t)m * m;
    const uint32_t Rh = (uint32_t)(r.R >> 32), Rl = (uint32_t)r.R, mh = (uint32_t)(mm >> 32), ml = (uint32_t)mm;
    // R m^2 2^-32 = 2^(300 - 2 E) (1 - e) modulo 2^64
    const uint64_t T = (uint64_t)Rh * ml + (((uint64_t)Rl * ml) >> 32) + (uint64_t)Rl * mh +
                       ((uint64_t)(uint32_t)(Rh * mh) << 32);
    const long long e60 = -(long long)T >> (240 - 2 * v.E);            // e in units of 2^-60
    const int e40 = (int)(e60 >> 20);
    const long long d60 = (e60 >> 1) + ((3 * (long long)e40 * e40) >> 23);
    v.M = ((uint64_t)m << 39) + (uint64_t)(((long long)m * d60) >> 21);
    v.x = v.E + r.s + k;
    return v;
}
__host__ __device__ __forceinline__ double fixed_ri(FixedInverse v) {
    const int z = lead_zeros32((uint32_t)(v.M >> 32) | 0x20000000u);   // 0..2
    return fixed_assemble(v.M, z, v.x - z + 848);
}
// 1/r^3 = M3 2^(3 x - 584), M3 in [2^59, 2^62]
__host__ __device__ __forceinline__ uint64_t fixed_cube(FixedInverse v) {
    const uint32_t h = (uint32_t)(v.M >> 32), l = (uint32_t)v.M;
    const uint64_t M2 = (((uint64_t)h * h) << 1) + (((uint64_t)h * l) >> 30);              // M^2 2^-63
    const uint32_t h2 = (uint32_t)(M2 >> 32), l2 = (uint32_t)M2;
    return (uint64_t)h * h2 + (((uint64_t)h * l2 + (uint64_t)l * h2) >> 32);
}

// A charge as mantissa and exponent: q = m 2^(e - 565), m in [2^62, 2^63), up to its sign; 0 has m = 0 and an
// empty mask.  false: no integer form (subnormal, or beyond 2^+-200, where products may leave float64's range).
struct FixedCharge {
    uint64_t m;
    int e;
    uint32_t keep;
};
__host__ __device__ __forceinline__ bool fixed_charge(double q, FixedCharge& c) {
    const uint64_t b = (uint64_t)f64_bits(q) & 0x7fffffffffffffffull;
    const int E = (int)(b >> 52);
    c.keep = b ? 0xffffffffu : 0u;
    c.m = b ? ((b << 10) & 0x3fffffffffffffffull) | (1ull << 62) : 0;
    c.e = b ? E - 520 : 0;
    return !b || (E >= 823 && E <= 1223);
}
// q / r^3 from the cube, rounded once
__host__ __device__ __forceinline__ double fixed_weight(uint64_t M3, int x3, FixedCharge c, double q) {
    const uint32_t h = (uint32_t)(M3 >> 32), l = (uint32_t)M3, H = (uint32_t)(c.m >> 32), L = (uint32_t)c.m;
    const uint64_t P = (uint64_t)h * H + (((uint64_t)h * L + (uint64_t)l * H) >> 32);      // 0 or in [2^57, 2^61)
    const int z = lead_zeros32((uint32_t)(P >> 32) | 0x01000000u);                         // 3..6
    const uint64_t mant = ((P >> (10 - z)) + 1) >> 1;
    const uint32_t hi = (uint32_t)(mant >> 32) + ((uint32_t)(x3 + c.e - z) << 20);
    return f64_from((long long)(((uint64_t)((hi & c.keep) | ((uint32_t)((uint64_t)f64_bits(q) >> 32) & 0x80000000u)) << 32) |
                                (uint32_t)mant));
}

}  // namespace psum
