// What the device headers under test need of CUDA, for a host compiler: the
// rounding intrinsics (IEEE operations of the host, contraction off), the
// bit casts, and one thread in place of the cooperative operations.
#pragma once
#include <cuda_runtime.h>

#include <algorithm>
#include <cfloat>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <vector>

using std::fabs;
using std::fmax;
using std::max;
using std::min;

#undef __noinline__
#define __noinline__ __attribute__((noinline))

template <class To, class From>
static inline To bits_of(From x) {
  static_assert(sizeof(To) == sizeof(From), "size");
  To r;
  std::memcpy(&r, &x, sizeof r);
  return r;
}

static inline float __fadd_rn(float a, float b) { return a + b; }
static inline float __fmul_rn(float a, float b) { return a * b; }
static inline float __fmaf_rn(float a, float b, float c) { return std::fmaf(a, b, c); }
static inline double __dadd_rn(double a, double b) { return a + b; }
static inline double __dmul_rn(double a, double b) { return a * b; }
static inline double __fma_rn(double a, double b, double c) { return std::fma(a, b, c); }
static inline double __ddiv_rn(double a, double b) { return a / b; }
static inline float2 __fadd2_rn(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
static inline float2 __fmul2_rn(float2 a, float2 b) { return make_float2(a.x * b.x, a.y * b.y); }
static inline float2 __ffma2_rn(float2 a, float2 b, float2 c) {
  return make_float2(std::fmaf(a.x, b.x, c.x), std::fmaf(a.y, b.y, c.y));
}
static inline float __fdividef(float a, float b) { return a / b; }
static inline double rsqrt(double x) { return 1.0 / std::sqrt(x); }
static inline float rsqrtf(float x) { return 1.0f / std::sqrt(x); }
static inline unsigned __float_as_uint(float a) { return bits_of<unsigned>(a); }
static inline float __uint_as_float(unsigned a) { return bits_of<float>(a); }
static inline float __int_as_float(int a) { return bits_of<float>(a); }
static inline int __double2hiint(double x) { return (int)(bits_of<uint64_t>(x) >> 32); }
static inline int __double2loint(double x) { return (int)bits_of<uint64_t>(x); }
static inline double __hiloint2double(int h, int l) {
  return bits_of<double>((uint64_t)(unsigned)h << 32 | (unsigned)l);
}
static inline double __longlong_as_double(long long v) { return bits_of<double>(v); }
static inline unsigned __funnelshift_l(unsigned lo, unsigned hi, int s) {
  return (hi << s) | (lo >> (32 - s));
}
static inline float __uint2float_rn(unsigned x) { return (float)x; }

struct HostIndex {
  unsigned x, y, z;
};
static HostIndex threadIdx, blockIdx, blockDim;
static inline void __syncthreads() {}
template <class T>
static inline T __shfl_sync(unsigned, T v, int) { return v; }
template <class T>
static inline T __shfl_xor_sync(unsigned, T v, int) { return v; }
static inline unsigned __reduce_max_sync(unsigned, unsigned v) { return v; }
template <class T>
static inline T atomicAdd(T* p, T v) { const T o = *p; *p += v; return o; }
template <class T>
static inline T atomicOr(T* p, T v) { const T o = *p; *p |= v; return o; }

// the one inline instruction of these headers on this path is rcp.approx
#define asm(...) (r = 1.0f / x)
