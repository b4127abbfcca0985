// dugks_sum.cuh -- sums of doubles as integers.
//
// The FP64 unit of a scheduler takes 64 cycles for a warp's addition, so a short sum by one CTA is mostly
// that. Here each value becomes an integer of 113 bits, aligned to the largest exponent; 2048 of
// them add up in 128 bits. Cut off is what lies below 2^-112 of the largest value, and the sum is rounded
// once: closer than any order of FP64 additions, and the same in every order.
#pragma once

#include <cstdint>
#include <cstring>

namespace dugks {

constexpr int SUM_MAX = 2048;                        // values
constexpr int SUM_LO = 256, SUM_HI = 2030;           // largest exponents (biased) that keep every exponent below normal

__host__ __device__ inline uint64_t double_bits(double v) {
#ifdef __CUDA_ARCH__
    return (uint64_t)__double_as_longlong(v);
#else
    uint64_t u;
    std::memcpy(&u, &v, sizeof u);
    return u;
#endif
}
__host__ __device__ inline double bits_double(uint64_t u) {
#ifdef __CUDA_ARCH__
    return __longlong_as_double((long long)u);
#else
    double v;
    std::memcpy(&v, &u, sizeof v);
    return v;
#endif
}
__host__ __device__ inline int exponent_of(double v) { return (int)(double_bits(v) >> 52) & 0x7ff; }

// v in units of 2^(top - 1135), rounded toward zero (0 for zero and subnormal numbers)
__host__ __device__ inline __int128 aligned(double v, int top) {
    const uint64_t u = double_bits(v);
    const int ex = (int)(u >> 52) & 0x7ff, d = top - ex;
    if (ex == 0 || d >= 113) return 0;
    const uint64_t m = (u & 0xfffffffffffffull) | 0x10000000000000ull;
    // m * 2^(60 - d)
    const __int128 a = d <= 60 ? (__int128)((unsigned __int128)m << (60 - d)) : (__int128)(m >> (d - 60));
    return (int64_t)u < 0 ? -a : a;
}

// the double nearest to s 2^(top - 1135)
__host__ __device__ inline double unaligned(__int128 s, int top) {
    if (s == 0) return 0.0;
    const bool neg = s < 0;
    const unsigned __int128 a = neg ? (unsigned __int128)(-s) : (unsigned __int128)s;
    const uint64_t hi = (uint64_t)(a >> 64), lo = (uint64_t)a;
#ifdef __CUDA_ARCH__
    const int z = hi ? __clzll((long long)hi) : 64 + __clzll((long long)lo);
#else
    const int z = hi ? __builtin_clzll(hi) : 64 + __builtin_clzll(lo);
#endif
    const unsigned __int128 n = a << z;   // the leading bit is bit 127, of weight 2^(127 - z)
    const uint64_t t = (uint64_t)(n >> 64);
    uint64_t m = t >> 11;                 // 53 bits; the rest decides the rounding, to even where it is a half
    const uint64_t r = t & 0x7ff;
    if (r > 0x400 || (r == 0x400 && ((uint64_t)n != 0 || (m & 1)))) m++;
    const int e = top - 1135 + 127 - z;   // m is 2^52 .. 2^53: value m 2^(e - 52)
    const uint64_t u = ((uint64_t)(e + 1022) << 52) + m;   // (m's leading bit adds one to the exponent)
    return bits_double(u | (neg ? 0x8000000000000000ull : 0));
}

}  // namespace dugks
