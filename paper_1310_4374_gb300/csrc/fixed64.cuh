// Float64 pair terms with their geometry in 64-bit integers.  The float64 pipe issues one warp instruction
// per scheduler in 64 cycles and bounds the float64 pair kernels, while the integer pipes beside it are idle.
// Coordinates are integers in units of 2^-k, 2^(62-k) being a power of two above every coordinate difference
// of the system (fixed_scale): differences are exact, the squared distance keeps 58 to 62 bits, and 1/r, 1/r^3
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

// x 2^k, rounded; beyond +-2^62 (and for NaN and infinities) +-2^62, which no pair in the range reaches
__host__ __device__ __forceinline__ long long to_fixed(double x, int k) {
    const long long b = f64_bits(x);
    const int e = (int)(b >> 52) & 0x7ff, s = e - 1075 + k;
    const long long m = e ? (b & 0xfffffffffffffll) | (1ll << 52) : 0;
    const long long v = s > 9 ? (m ? 1ll << 62 : 0) : s >= 0 ? m << s : s > -54 ? (m + (1ll << (-s - 1))) >> -s : 0;
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
// square of its low word, 3 units of R together.
struct FixedR2 {
    uint64_t R;
    int s;
};
__host__ __device__ __forceinline__ FixedR2 fixed_r2(FixedDelta x, FixedDelta y, FixedDelta z, uint32_t high) {
    FixedR2 r;
    r.s = lead_zeros32(high) - 2;
    const uint64_t a = x.a << r.s, b = y.a << r.s, c = z.a << r.s;
    const uint32_t ah = (uint32_t)(a >> 32), bh = (uint32_t)(b >> 32), ch = (uint32_t)(c >> 32);
    const uint64_t cross = (uint64_t)ah * (uint32_t)a + (uint64_t)bh * (uint32_t)b + (uint64_t)ch * (uint32_t)c;
    r.R = (uint64_t)ah * ah + (uint64_t)bh * bh + (uint64_t)ch * ch + (cross >> 31);
    return r;
}
// The float32 copy of R 2^-32 for the estimate of its inverse square root.
__host__ __device__ __forceinline__ float fixed_estimate_arg(uint64_t R) { return (float)(uint32_t)(R >> 32); }

// mantissa M (leading one in bit 63 - z) times 2^(x - 1) with bit 52 as the unit, rounded
__host__ __device__ __forceinline__ double fixed_assemble(uint64_t M, int z, int x) {
    const uint64_t mant = ((M >> (10 - z)) + 1) >> 1;
    return f64_from((long long)(mant + ((uint64_t)(uint32_t)x << 52)));
}

// 1/r and 1/r^3 from the bits yb of a float32 estimate y of (R 2^-32)^(-1/2), relative error below 2^-21:
// with e = 1 - R 2^-32 y^2 (its integer is minus the product's low 64 bits, the leading one cancelling),
//   (R 2^-32)^(-1/2) = y (1 + e/2 + (3/8) e^2) + O((5/16) e^3), the rest below 2^-64;
// the cube from its 62-bit mantissa.  Errors before the rounding to 53 bits: 2^-57 and 2^-55.
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
    const int z = lead_zeros32((uint32_t)(v.M >> 32));                 // 0..2
    return fixed_assemble(v.M, z, v.x - z + 848);
}
__host__ __device__ __forceinline__ double fixed_ri3(FixedInverse v) {
    const uint32_t h = (uint32_t)(v.M >> 32), l = (uint32_t)v.M;
    const uint64_t M2 = (uint64_t)h * h + (((uint64_t)h * l) >> 31);   // M^2 2^-64
    const uint32_t h2 = (uint32_t)(M2 >> 32), l2 = (uint32_t)M2;
    const uint64_t M3 = (uint64_t)h * h2 + (((uint64_t)h * l2 + (uint64_t)l * h2) >> 32);
    const int z = lead_zeros32((uint32_t)(M3 >> 32));                  // 2..5
    return fixed_assemble(M3, z, 3 * v.x - z + 502);
}

}  // namespace psum
