// Host stand-ins for the CUDA built-ins that the device headers use, so that their per-cell functions
// compile with a C++ compiler and run on the CPU, one "thread" at a time.  Rounded operations are the
// plain ones (compile with -ffp-contract=off); library functions are the host's.
#pragma once
#include <cuda_runtime.h>
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>

using std::isfinite;
using std::max;
using std::min;

#undef __forceinline__
#define __forceinline__ inline
#undef __noinline__
#define __noinline__
#undef __launch_bounds__
#define __launch_bounds__(...)
#undef __grid_constant__
#define __grid_constant__

static const uint3 threadIdx{}, blockIdx{};
static const dim3 blockDim(1), gridDim(1);

template <class T, class U>
static inline T host_bits(U u) {
    static_assert(sizeof(T) == sizeof(U), "size");
    T t;
    std::memcpy(&t, &u, sizeof t);
    return t;
}
static inline unsigned __float_as_uint(float f) { return host_bits<unsigned>(f); }
static inline int __float_as_int(float f) { return host_bits<int>(f); }
static inline float __uint_as_float(unsigned u) { return host_bits<float>(u); }
static inline float __int_as_float(int i) { return host_bits<float>(i); }
static inline long long __double_as_longlong(double d) { return host_bits<long long>(d); }
static inline double __longlong_as_double(long long i) { return host_bits<double>(i); }
static inline int __double2hiint(double d) { return (int)(host_bits<uint64_t>(d) >> 32); }
static inline int __double2loint(double d) { return (int)(unsigned)host_bits<uint64_t>(d); }
static inline double __hiloint2double(int h, int l) {
    return host_bits<double>(((uint64_t)(unsigned)h << 32) | (uint64_t)(unsigned)l);
}
static inline unsigned __funnelshift_l(unsigned lo, unsigned hi, unsigned s) {
    return (unsigned)(((((uint64_t)hi << 32) | lo) << (s & 31)) >> 32);
}
static inline unsigned long long __umul64hi(unsigned long long a, unsigned long long b) {
    return (unsigned long long)(((unsigned __int128)a * b) >> 64);
}
static inline unsigned __umulhi(unsigned a, unsigned b) { return (unsigned)(((uint64_t)a * b) >> 32); }
static inline double __dadd_rn(double a, double b) { return a + b; }
static inline double __dsub_rn(double a, double b) { return a - b; }
static inline double __dmul_rn(double a, double b) { return a * b; }
static inline double __ddiv_rn(double a, double b) { return a / b; }
static inline double __fma_rn(double a, double b, double c) { return std::fma(a, b, c); }
static inline float __fadd_rn(float a, float b) { return a + b; }
static inline float __fsub_rn(float a, float b) { return a - b; }
static inline float __fmul_rn(float a, float b) { return a * b; }
static inline float __fmaf_rn(float a, float b, float c) { return std::fma(a, b, c); }
static inline float __fdividef(float a, float b) { return a / b; }
// as the device computes it: the rounded product with log2(e) costs |x| 2^-24 of the result
#define __expf(x) std::exp2((x) * 1.4426950408889634f)
template <class T>
static inline T __ldg(const T* p) { return *p; }
template <class T, class U>
static inline T atomicAdd(T* p, U v) { const T o = *p; *p = o + (T)v; return o; }
template <class T, class U>
static inline T atomicMax(T* p, U v) { const T o = *p; if ((T)v > o) *p = (T)v; return o; }
template <class T, class U>
static inline T atomicMin(T* p, U v) { const T o = *p; if ((T)v < o) *p = (T)v; return o; }
template <class T>
static inline T __shfl_xor_sync(unsigned, T v, int) { return v; }
template <class T>
static inline T __shfl_sync(unsigned, T v, int) { return v; }
static inline int __any_sync(unsigned, int p) { return p != 0; }
static inline void __syncthreads() {}
static inline void __syncwarp() {}
// named by code that no host check calls
static inline size_t __cvta_generic_to_shared(const void* p) { return (size_t)p; }
static inline __nv_bfloat162 __hfma2(__nv_bfloat162 a, __nv_bfloat162, __nv_bfloat162) { return a; }
