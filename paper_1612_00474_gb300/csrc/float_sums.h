// float_sums.h -- the end of a compensated float32 sum (no CUDA calls, so that the tests can compile and check it on
// the CPU).
#pragma once

#include <cstdint>
#include <cstring>

#ifndef RPB_HD
#ifdef __CUDACC__
#define RPB_HD __host__ __device__
#else
#define RPB_HD
#endif
#endif

namespace rpb {

// s += x, returning what float32 drops (Knuth's two-sum, exact).
RPB_HD inline float two_sum(float &s, float x)
{
    const float t = s + x, z = t - s;
    const float e = (s - (t - z)) + (x - z);
    s = t;
    return e;
}

// (double)x in integer instructions: a conversion holds its scheduler as long as a float64 addition does.
RPB_HD inline double widen(float x)
{
    uint32_t b;
    std::memcpy(&b, &x, sizeof b);
    const bool small = (b & 0x7fffffffu) < 0x00800000u;  // zero or not normal: scaled by 2^64
    const float y = small ? x * 18446744073709551616.f : x;
    std::memcpy(&b, &y, sizeof b);
    const uint32_t m = b & 0x7fffffffu;
    // the exponents' biases differ by 896; that of infinities and NaN goes from 255 to 2047
    const uint32_t bias = m >= 0x7f800000u ? 2u * 896u : (small ? 896u - 64u : 896u);
    const uint64_t v = m == 0u ? 0u : ((uint64_t)m << 29) + ((uint64_t)bias << 52);
    const uint64_t d = v | (uint64_t)(b & 0x80000000u) << 32;
    double r;
    std::memcpy(&r, &d, sizeof r);
    return r;
}

// A sum of float32 numbers good to float64's rounding: in float32, as a sum, the exact errors of its additions, and the
// errors of those additions, whose own rounding is 2^-70 of the largest number.  One conversion and two additions in
// float64 in all, instead of one of each for every number (a float64 warp instruction takes 64 cycles of its
// scheduler).
struct FloatSum {
    float hi, lo, rest;
    RPB_HD void add_low(float x) { rest += two_sum(lo, x); }
    RPB_HD void add(float x) { add_low(two_sum(hi, x)); }
    RPB_HD void add(const FloatSum &o)
    {
        add(o.hi);
        add_low(o.lo);
        rest += o.rest;
    }
    RPB_HD double value() const { return (double)hi + (widen(lo) + widen(rest)); }
};

// sum over u of s[u] - c[u]: four compensated (Kahan) chains and their corrections
RPB_HD inline FloatSum join_sums(const float (&s)[4], const float (&c)[4])
{
    FloatSum f = {s[0], -c[0], 0.f};
#ifdef __CUDACC__
#pragma unroll
#endif
    for (int u = 1; u < 4; ++u) {
        f.add(s[u]);
        f.add_low(-c[u]);
    }
    return f;
}

}  // namespace rpb
