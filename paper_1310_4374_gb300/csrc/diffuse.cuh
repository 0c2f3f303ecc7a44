// The float32 rounding of a group's charges with the error carried along the group, as integers
// (the pack kernel's chain; sort.cu says why it exists and what it costs).
#pragma once

#include <stdint.h>
#include <string.h>

namespace psum {

constexpr int kQBits = 62;                               // fixed-point charges: |Q| < 2^kQBits
constexpr int kExpLo = 1023 - 60, kExpHi = 1023 + 126;   // largest biased exponents the chain takes

// the biased exponent field of a double's bits
__host__ __device__ __forceinline__ int exp_field(long long bits) { return (int)((bits >> 52) & 0x7ff); }

// A finite double (by its bits) as a fixed-point integer in units of 2^(emax - 1022 - kQBits), where
// emax is the largest biased exponent of the group: exact down to 2^-9 of the largest charge, below
// that rounded to the unit.
__host__ __device__ __forceinline__ long long fixed_charge(long long bits, int emax) {
    const int e = exp_field(bits);
    long long m = (bits & 0xfffffffffffffll) | (e ? 1ll << 52 : 0ll);
    const int sh = (kQBits - 53) - (emax - (e ? e : 1));
    if (sh >= 0)
        m <<= sh;
    else
        m = -sh > 54 ? 0ll : (m + (1ll << (-sh - 1))) >> -sh;
    return bits < 0 ? -m : m;
}
__host__ __device__ __forceinline__ double fixed_unit(int emax) {
    const long long b = (long long)(emax - 1022 - kQBits + 1023) << 52;
    double u;
    memcpy(&u, &b, sizeof u);
    return u;
}

// bits of v below the 24 that a float32 keeps
__host__ __device__ __forceinline__ int dropped_bits(long long v) {
    const unsigned long long a = v < 0 ? 0ull - (unsigned long long)v : (unsigned long long)v;
#ifdef __CUDA_ARCH__
    const int n = 40 - __clzll((long long)a);
#else
    const int n = a ? 40 - __builtin_clzll(a) : 0;
#endif
    return n > 0 ? n : 0;
}

// One step of the chain: the carry out of a charge with its half unit in the last kept place
// already added (Uh = Q + (mask + 1)/2) and the carry c coming in.
__host__ __device__ __forceinline__ long long diffuse_step(long long Uh, long long mask, long long c) {
    return ((mask + 1) >> 1) - ((Uh - c) & mask);
}

// The rounded charge of Q with carry c coming in, and whether the chain's assumptions hold for it:
// Q - c still drops the bits that Q does, and its rounding is no tie.
__host__ __device__ __forceinline__ long long diffuse_value(long long Q, long long c, bool& fine) {
    const int d = dropped_bits(Q);
    const long long mask = (1ll << d) - 1, T = Q - c, U = T + ((mask + 1) >> 1);
    fine = dropped_bits(T) == d && !(d && (U & mask) == 0);
    return U & ~mask;
}

}  // namespace psum
