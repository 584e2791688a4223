// Host stand-ins for the CUDA names the relativistic recovery's headers use, so
// that its arithmetic can be compiled and checked by the host compiler.
#pragma once
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>
#define __device__
#define __host__
#define __forceinline__ inline
#define __noinline__
using std::fabs;
using std::fmax;
using std::fmin;
using std::isfinite;
using std::max;
using std::min;
inline float __fadd_rn(float a, float b) { return a + b; }
inline float __fmul_rn(float a, float b) { return a * b; }
inline float __fmaf_rn(float a, float b, float c) { return std::fmaf(a, b, c); }
#ifdef SEED_ULPS  // the approximate forms, up to that many units in the last place off
inline float ulps_off(float r)
{
    uint32_t u;
    std::memcpy(&u, &r, 4);
    if ((u & 0x7F800000u) == 0u || (u & 0x7F800000u) == 0x7F800000u) return r;
    u += (u * 0x9E3779B9u >> 16) % (2 * SEED_ULPS + 1) - SEED_ULPS;
    std::memcpy(&r, &u, 4);
    return r;
}
#else
inline float ulps_off(float r) { return r; }
#endif
inline float __fdividef(float a, float b) { return ulps_off(a / b); }
inline float rsqrtf(float x) { return ulps_off((float)(1.0 / std::sqrt((double)x))); }
template <class T, class F> inline T bits_as(F f)
{
    T t;
    static_assert(sizeof(T) == sizeof(F), "same size");
    std::memcpy(&t, &f, sizeof(T));
    return t;
}
inline int __double2hiint(double x) { return (int)(bits_as<uint64_t>(x) >> 32); }
inline int __double2loint(double x) { return (int)(uint32_t)bits_as<uint64_t>(x); }
inline double __hiloint2double(int h, int l) { return bits_as<double>(((uint64_t)(uint32_t)h << 32) | (uint32_t)l); }
inline float __uint_as_float(unsigned u) { return bits_as<float>(u); }
inline unsigned __float_as_uint(float f) { return bits_as<unsigned>(f); }
inline long long __double_as_longlong(double d) { return bits_as<long long>(d); }
inline double __longlong_as_double(long long u) { return bits_as<double>(u); }
// float64 seeds like the hardware's approximations: about 2^-23 and 2^-22 off,
// results and arguments below the normal range zero
namespace ctu {
inline double seed_off(double r, double rel)
{
    const uint64_t h = bits_as<uint64_t>(r) * 0x9E3779B97F4A7C15ull;
    r *= 1.0 + rel * ((double)(h >> 40) / 8388608.0 - 1.0);
    return std::fabs(r) < 2.2250738585072014e-308 ? std::copysign(0.0, r) : r;
}
inline double seed_arg(double x) { return std::fabs(x) < 2.2250738585072014e-308 ? std::copysign(0.0, x) : x; }
inline double d_rcp_seed(double x) { return seed_off(1.0 / seed_arg(x), 1.19e-7); }
inline double d_rsqrt_seed(double x) { return seed_off(1.0 / std::sqrt(seed_arg(x)), 2.38e-7); }
} // namespace ctu
