// The device headers (csrc/*.cuh) compiled as plain C++ for a CPU test: the qualifiers and the
// intrinsics they use, with the rounding of the device forms (build with -ffp-contract=off).
// rsqrtf and __fdividef are the correctly rounded forms here.
#pragma once
#define __device__
#define __host__
#define __global__
#define __forceinline__ inline
#define __noinline__ __attribute__((noinline))
#define __launch_bounds__(...)
#define __grid_constant__
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>
using std::isfinite;
using std::max;
using std::min;
template <class To, class From>
inline To bits_as(From v)
{
    To r;
    static_assert(sizeof r == sizeof v, "");
    std::memcpy(&r, &v, sizeof r);
    return r;
}
inline int __double2hiint(double x) { return (int)(bits_as<uint64_t>(x) >> 32); }
inline int __double2loint(double x) { return (int)(uint32_t)bits_as<uint64_t>(x); }
inline double __hiloint2double(int hi, int lo) { return bits_as<double>((uint64_t)(uint32_t)hi << 32 | (uint32_t)lo); }
inline long long __double_as_longlong(double x) { return bits_as<long long>(x); }
inline double __longlong_as_double(long long b) { return bits_as<double>(b); }
inline float __uint_as_float(unsigned b) { return bits_as<float>(b); }
inline float __int_as_float(int b) { return bits_as<float>(b); }
inline unsigned __float_as_uint(float x) { return bits_as<unsigned>(x); }
inline int __float_as_int(float x) { return bits_as<int>(x); }
inline float __fadd_rn(float a, float b) { return a + b; }
inline float __fsub_rn(float a, float b) { return a - b; }
inline float __fmul_rn(float a, float b) { return a * b; }
inline float __fsqrt_rn(float a) { return std::sqrt(a); }
inline float __frcp_rn(float a) { return 1.0f / a; }
inline float __fdividef(float a, float b) { return std::fabs(b) > 0x1p126f && std::fabs(b) < INFINITY ? 0.0f * a : a / b; }
inline float rsqrtf(float a) { return (float)(1.0 / std::sqrt((double)a)); }
inline double rsqrt(double a) { return 1.0 / std::sqrt(a); }
inline unsigned __umulhi(unsigned a, unsigned b) { return (unsigned)((uint64_t)a * b >> 32); }
template <class T> inline T atomicAdd(T* p, T v) { T o = *p; *p += v; return o; }
struct Idx3 { unsigned x, y, z; };
inline thread_local Idx3 threadIdx{0, 0, 0}, blockIdx{0, 0, 0}, blockDim{1, 1, 1}, gridDim{1, 1, 1};
