// The CUDA built-ins that the device headers use, as plain C++, so that the
// searches can be compiled and compared with one another on the CPU.
#pragma once
#include <cmath>
#include <cstdint>
#include <cstring>

#include <cuda_runtime.h>

using std::abs;
using std::isfinite;
using std::max;
using std::min;

#undef __forceinline__
#define __forceinline__ inline

template <typename T, typename F>
static inline T bits_as(F x)
{
    static_assert(sizeof(T) == sizeof(F), "bits_as");
    T y;
    memcpy(&y, &x, sizeof y);
    return y;
}
static inline float __int_as_float(int x) { return bits_as<float>(x); }
static inline unsigned __float_as_uint(float x) { return bits_as<unsigned>(x); }
static inline double __longlong_as_double(long long x) { return bits_as<double>(x); }
static inline long long __double_as_longlong(double x) { return bits_as<long long>(x); }
static inline int __double2hiint(double x) { return (int)(bits_as<unsigned long long>(x) >> 32); }
static inline double __hiloint2double(int hi, int lo)
{
    return bits_as<double>((unsigned long long)(unsigned)hi << 32 | (unsigned)lo);
}
static inline float __fdividef(float a, float b) { return a / b; }
static inline float __frcp_rn(float x) { return 1.0f / x; }
static inline double __drcp_rn(double x) { return 1.0 / x; }
static inline float __fmul_rn(float a, float b) { return a * b; }
static inline double __dmul_rn(double a, double b) { return a * b; }
static inline float __fadd_rn(float a, float b) { return a + b; }
static inline double __dadd_rn(double a, double b) { return a + b; }
static inline float __fmaf_rn(float a, float b, float c) { return fmaf(a, b, c); }
static inline double __fma_rn(double a, double b, double c) { return fma(a, b, c); }
static inline unsigned __umulhi(unsigned a, unsigned b) { return (unsigned)((unsigned long long)a * b >> 32); }
static inline unsigned __float2uint_rn(float x) { return (unsigned)rintf(x); }
template <typename T>
static inline T __ldg(const T* p) { return *p; }
static const dim3 threadIdx(0, 0, 0), blockDim(1, 1, 1);
