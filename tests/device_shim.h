// Host definitions of the CUDA intrinsics and built-in variables that csrc/gdg_internal.cuh uses, so that its device functions
// compile as host C++ (one thread).
#pragma once
#include <cuda_runtime.h>
#include <math.h>
#include <string.h>
#include <algorithm>
#define __noinline__ __attribute__((noinline))
template <class T, class F> static inline T bits_as(F f) { T t; memcpy(&t, &f, sizeof t); return t; }
static inline double __longlong_as_double(long long x) { return bits_as<double>(x); }
static inline long long __double_as_longlong(double x) { return bits_as<long long>(x); }
static inline int __double2hiint(double x) { return (int)(bits_as<unsigned long long>(x) >> 32); }
static inline int __double2loint(double x) { return (int)bits_as<unsigned long long>(x); }
static inline double __hiloint2double(int h, int l) { return bits_as<double>(((unsigned long long)(unsigned)h << 32) | (unsigned)l); }
static inline float __uint_as_float(unsigned x) { return bits_as<float>(x); }
static inline unsigned __float_as_uint(float x) { return bits_as<unsigned>(x); }
static inline double __dmul_rn(double a, double b) { return a * b; }
static inline float __fmul_rn(float a, float b) { return a * b; }
static inline float __fadd_rn(float a, float b) { return a + b; }
static inline float __fdiv_rn(float a, float b) { return a / b; }
static inline float __frcp_rn(float a) { return 1.0f / a; }
static inline unsigned __activemask() { return 1u; }
static inline int __ffs(int) { return 1; }
static inline int __popc(unsigned) { return 1; }
static inline unsigned __shfl_sync(unsigned, unsigned v, int) { return v; }
static inline unsigned atomicAdd(unsigned* p, unsigned v) { unsigned o = *p; *p += v; return o; }
static uint3 threadIdx, blockIdx;
static dim3 blockDim, gridDim;
static inline void __syncthreads() {}
template <class T> static inline T __ldg(const T* p) { return *p; }
