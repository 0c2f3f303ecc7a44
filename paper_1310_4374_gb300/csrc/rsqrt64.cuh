// Float64 1/r and 1/r^3 from a float32 estimate, with as few float64 operations as they need: the
// float64 pipe (one warp instruction per scheduler in 64 cycles, conversions included) bounds the
// float64 pair kernels, the integer and float32 pipes beside it are idle.  The form of the pairs that the
// integer coordinates leave out (fixed64.cuh).
#pragma once

#include <math.h>
#include <stdint.h>
#include <string.h>

namespace psum {

__host__ __device__ __forceinline__ long long f64_bits(double x) {
    long long b;
    memcpy(&b, &x, sizeof b);
    return b;
}
__host__ __device__ __forceinline__ double f64_from(long long b) {
    double x;
    memcpy(&x, &b, sizeof x);
    return x;
}
__host__ __device__ __forceinline__ float f32_from(uint32_t b) {
    float x;
    memcpy(&x, &b, sizeof x);
    return x;
}
__host__ __device__ __forceinline__ int lead_zeros32(uint32_t v) {
#ifdef __CUDA_ARCH__
    return __clz((int)v);
#else
    return v ? __builtin_clz(v) : 32;
#endif
}
__host__ __device__ __forceinline__ uint32_t round_u32(float v) {
#ifdef __CUDA_ARCH__
    return __float2uint_rn(v);
#else
    return (uint32_t)nearbyintf(v);
#endif
}

// The float32 copy of r2 for the estimate: the exponent rebiased (1023 -> 127) and the mantissa cut to
// 23 bits, on the bits; 0 below 2^-126, which would need two charges within 1e-19 of each other.
__host__ __device__ __forceinline__ float estimate_arg(double r2) {
    const long long t = (f64_bits(r2) >> 29) - (896LL << 23);
    return f32_from(t >= 1LL << 23 ? (uint32_t)t : 0u);
}
// 1/r^3 where that copy is 0: charges within 2^-63.5 count as coincident, K(0) = 0; up to 2^-63 the pair is out of
// the form's range, and an infinite field has the evaluation refused as not finite.
__host__ __device__ __forceinline__ double rsqrt3_below(double r2) {
    const long long t = (f64_bits(r2) >> 29) - (896LL << 23);
    return f64_from(t > 0 && t < 1LL << 23 ? 0x7ffLL << 52 : 0LL);
}
// The magnitude of a float64 below 1 as float32, 20 mantissa bits; 0 below 2^-100.
__host__ __device__ __forceinline__ float small_magnitude(double e) {
    const int ea = (int)(f64_bits(e) >> 32) & 0x7fffffff;
    return f32_from(ea > (923 << 20) ? (uint32_t)(ea - (896 << 20)) << 3 : 0u);
}

// 1/sqrt(r2) from the bits yb of a float32 estimate y of it (relative error below 2^-22, of r2's
// float32 copy): with e = 1 - r2 y^2, |e| < 2^-21,
//   1/sqrt(r2) = y (1 - e)^(-1/2) = y + (y/2)(e + (3/4) e^2) + O(y e^3),
// the rest (5/16)|e|^3 < 1e-19 being below float64 rounding.  y^2 is the exact 48-bit square of y's
// 24-bit mantissa, an integer product put back under its exponent, and the factor 3/4 e needs 10 bits:
// it is float32, widened.  Three float64 operations (e, its square's term, the final multiply-add)
// where the estimate's square, the series and its products took five.
__host__ __device__ __forceinline__ double rsqrt_refined(double r2, uint32_t yb) {
    // float64 bits of the (positive, normal) estimate: exponent rebiased, mantissa widened
    const long long yw = ((long long)yb << 29) + (896LL << 52);
    // y^2 = 2^(2 E) (m / 2^23)^2 with m in [2^23, 2^24): a product of 47 or 48 bits, whose leading
    // one, shifted to bit 52, adds itself to the exponent below it
    const uint32_t m = (yb & 0x7fffffu) | 0x800000u;
    const uint64_t mm = (uint64_t)m * m;
    const int top = (int)(mm >> 47);                                   // 1: (m / 2^23)^2 >= 2
    const long long ex = 2 * (long long)(yb >> 23) - 254 + 1022 + top;
    const double yy = f64_from((ex << 52) + (long long)(mm << (6 - top)));
    const double e = fma(-r2, yy, 1.0);
    const float ge = 0.75f * small_magnitude(e);
    uint32_t gb;
    memcpy(&gb, &ge, sizeof gb);
    const long long g = ((long long)gb << 29) + (gb ? 896LL << 52 : 0LL);
    const double es = f64_from(g | (f64_bits(e) & (long long)0x8000000000000000ull));
    return fma(f64_from(yw - (1LL << 52)), fma(es, e, e), f64_from(yw));
}

// r2^(-3/2) from the same estimate, for the pair terms of potential and field together (q r^-3 times
// the offset, and times r2 for the potential):
//   r2^(-3/2) = y^3 (1 - e)^(-3/2) = y^3 (1 + (3/2) e + (15/8) e^2) + O(y^3 e^3), 35/16 |e|^3 < 2^-61.
// y^3 is a 72-bit integer product; its second-order term (at most 2^-41 of it, from float32) joins it
// before its one rounding to 53 bits; 3/2 e is formed as such, (3/2) y^2 being an exact 50-bit integer.
// Two float64 operations where 1/r, its square and its cube took five, and two roundings (at most one
// unit in the last place together) where the cube tripled the error of 1/r.
__host__ __device__ __forceinline__ double rsqrt3_refined(double r2, uint32_t yb) {
    const int E = (int)(yb >> 23);                                     // y = m 2^(E - 150), m in [2^23, 2^24)
    const uint32_t m = (yb & 0x7fffffu) | 0x800000u;
    const uint64_t mm = (uint64_t)m * m, mm3 = 3 * mm;                 // mm3 in [2^47, 2^50)
    const int s2 = lead_zeros32((uint32_t)(mm3 >> 32)) - 11;           // 3..5: its leading one to bit 52
    const double e = fma(-r2, f64_from(((long long)(2 * E + 773 - s2) << 52) + (long long)(mm3 << s2)), 1.5);
    // y^3 = V 2^(3E - 442), V = m^3 / 2^8 in [2^61, 2^64); (15/8)(2/3)^2 e^2 of it in units of V
    const float ef = small_magnitude(e), mf = f32_from((yb & 0x7fffffu) | 0x3f800000u);   // mf = m / 2^23
    const uint32_t second = round_u32(ef * ef * (mf * mf) * (mf * 1.9215358e18f));         // 5/6 * 2^61
    const uint64_t lo = (uint64_t)(uint32_t)mm * m;
    const uint64_t up = (uint64_t)(uint32_t)(mm >> 32) * m + (lo >> 32);                   // m^3 = up 2^32 + low word of lo
    const uint64_t V = (up << 24) + ((uint32_t)lo >> 8) + second;
    const int s3 = 11 - lead_zeros32((uint32_t)(V >> 32));             // 9..11 bits to drop
    const uint64_t mant = (V + (1ull << (s3 - 1))) >> s3;              // [2^52, 2^53]
    const double y3 = f64_from(((long long)(3 * E + 632 + s3) << 52) + (long long)mant);
    return fma(y3, e, y3);
}

}  // namespace psum
