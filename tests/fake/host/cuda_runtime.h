// enough of the CUDA language for a host compiler to build df.cuh: the intrinsics are single IEEE-754 operations
// (compile with -ffp-contract=off)
#pragma once
#include <math.h>
#include <string.h>

#define __device__
#define __forceinline__ inline
inline float __fadd_rn(float a, float b) { return a + b; }
inline float __fsub_rn(float a, float b) { return a - b; }
inline float __fmul_rn(float a, float b) { return a * b; }
inline float __fmaf_rn(float a, float b, float c) { return fmaf(a, b, c); }
inline float __int2float_rn(int i) { return (float)i; }
inline float rsqrtf(float x) { return 1.0f / sqrtf(x); }
template <typename To, typename From> inline To bits(From f) { To t; memcpy(&t, &f, sizeof t); return t; }
inline long long __double_as_longlong(double x) { return bits<long long>(x); }
inline double __longlong_as_double(long long x) { return bits<double>(x); }
inline unsigned __float_as_uint(float x) { return bits<unsigned>(x); }
inline float __uint_as_float(unsigned x) { return bits<float>(x); }
