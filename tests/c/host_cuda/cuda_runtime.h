/* Host stand-ins for the CUDA names that pp_arith.cuh and pp_hx.cuh use, so that a plain C++ compiler can run
 * their arithmetic (compile with -ffp-contract=off).  Integer sums go through the compiler's own checks. */
#pragma once
#include <cmath>
#include <cstring>
#define __device__
#define __host__
#define __forceinline__ inline
#define __noinline__
#define __align__(n) alignas(n)
struct float2 { float x, y; };
struct float4 { float x, y, z, w; };
struct double2 { double x, y; };
inline float2 make_float2(float x, float y) { return float2{x, y}; }
template <class T, class F> inline T bits_as(F v) { T r; static_assert(sizeof(T) == sizeof(F), ""); memcpy(&r, &v, sizeof r); return r; }
inline float __fadd_rn(float a, float b) { return a + b; }
inline float __fsub_rn(float a, float b) { return a - b; }
inline float __fmul_rn(float a, float b) { return a * b; }
inline float __fmaf_rn(float a, float b, float c) { return std::fma(a, b, c); }
inline float __frcp_rn(float a) { return 1.0f / a; }
inline double __dadd_rn(double a, double b) { return a + b; }
inline double __dmul_rn(double a, double b) { return a * b; }
inline double __ll2double_rn(long long a) { return (double)a; }
inline float __double2float_rn(double a) { return (float)a; }
inline float __int2float_rn(int a) { return (float)a; }
inline int __float2int_rn(float a) { return a != a ? 0 : a >= 2147483648.0f ? 2147483647 : a <= -2147483648.0f ? (-2147483647 - 1) : (int)std::nearbyint(a); }
inline int __clz(int a) { return a ? __builtin_clz((unsigned)a) : 32; }
inline unsigned __funnelshift_l(unsigned lo, unsigned hi, unsigned s) { return (unsigned)(((((unsigned long long)hi << 32) | lo) << (s & 31)) >> 32); }
inline int __double2hiint(double d) { return (int)(bits_as<unsigned long long>(d) >> 32); }
inline int __double2loint(double d) { return (int)(unsigned)bits_as<unsigned long long>(d); }
inline double __hiloint2double(int h, int l) { return bits_as<double>(((unsigned long long)(unsigned)h << 32) | (unsigned)l); }
inline long long __double_as_longlong(double d) { return bits_as<long long>(d); }
inline double __longlong_as_double(long long v) { return bits_as<double>(v); }
inline unsigned __float_as_uint(float f) { return bits_as<unsigned>(f); }
inline float __uint_as_float(unsigned u) { return bits_as<float>(u); }
inline int __float_as_int(float f) { return bits_as<int>(f); }
template <class T> inline T __ldg(const T* p) { return *p; }
