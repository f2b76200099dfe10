// Pairs of FP32 numbers as one value h + l ("double-float" arithmetic after
// Dekker, "A floating-point technique for extending the available
// precision", Numer. Math. 18, 1971, and Knuth's two-sum), about 48 bits.
//
// Why: one FP64 warp instruction occupies a GB300 sub-partition's FP64 pipe
// for 65 to 77 cycles (measured; DFMA 64.7, DADD and DMUL 76.6), one FP32 or
// logic instruction for 1 (FFMA 1.03, LOP3 0.85, IADD 1.09). A double-float
// sum is 11 FP32 instructions and a product 7, so the parts of the scheme
// that are a small correction to an FP64 result run here, next to the FP64
// pipe instead of on it. What may be computed in this form, and how its
// error compares with FP64, is stated where it is used (weno_df.cuh).
//
// Every operation is written with the _rn intrinsics, which the compiler
// neither contracts nor reorders.
#pragma once

#include <cuda_runtime.h>

namespace hweno {

struct D2 {
  float h, l;
};

// x (exactly representable constants and others) as a pair, at compile time.
__host__ __device__ constexpr D2 dconst(double x) {
  return D2{(float)x, (float)(x - (double)(float)x)};
}

__device__ __forceinline__ D2 renorm(float s, float e) {  // |e| <= |s|
  const float h = __fadd_rn(s, e);
  return D2{h, __fadd_rn(e, -__fadd_rn(h, -s))};
}
__device__ __forceinline__ D2 neg(D2 a) { return D2{-a.h, -a.l}; }
// a + b; the error is at most 2^-46 of |a| + |b| (differences included)
__device__ __forceinline__ D2 add(D2 a, D2 b) {
  const float s = __fadd_rn(a.h, b.h);
  const float t = __fadd_rn(s, -a.h);
  const float e = __fadd_rn(__fadd_rn(a.h, -__fadd_rn(s, -t)), __fadd_rn(b.h, -t));
  return renorm(s, __fadd_rn(e, __fadd_rn(a.l, b.l)));
}
__device__ __forceinline__ D2 sub(D2 a, D2 b) { return add(a, neg(b)); }
__device__ __forceinline__ D2 mul(D2 a, D2 b) {
  const float p = __fmul_rn(a.h, b.h);
  float e = __fmaf_rn(a.h, b.h, -p);
  e = __fmaf_rn(a.h, b.l, e);
  e = __fmaf_rn(a.l, b.h, e);
  return renorm(p, e);
}
__device__ __forceinline__ D2 mul(D2 a, float c) {
  const float p = __fmul_rn(a.h, c);
  return renorm(p, __fmaf_rn(a.l, c, __fmaf_rn(a.h, c, -p)));
}
__device__ __forceinline__ D2 square(D2 a) {
  const float p = __fmul_rn(a.h, a.h);
  return renorm(p, __fmaf_rn(__fadd_rn(a.h, a.h), a.l, __fmaf_rn(a.h, a.h, -p)));
}
// a times a power of two (exact)
__device__ __forceinline__ D2 scale(D2 a, float p2) {
  return D2{__fmul_rn(a.h, p2), __fmul_rn(a.l, p2)};
}
__device__ __forceinline__ D2 abs2(D2 a) { return a.h < 0.f ? neg(a) : a; }

// a * b + c without the intermediate renormalisation
__device__ __forceinline__ D2 madd(D2 a, D2 b, D2 c) {
  const float p = __fmul_rn(a.h, b.h);
  float e = __fmaf_rn(a.h, b.h, -p);
  e = __fmaf_rn(a.h, b.l, e);
  e = __fmaf_rn(a.l, b.h, e);
  const float s = __fadd_rn(p, c.h);
  const float t = __fadd_rn(s, -p);
  const float r = __fadd_rn(__fadd_rn(p, -__fadd_rn(s, -t)), __fadd_rn(c.h, -t));
  return renorm(s, __fadd_rn(r, __fadd_rn(e, c.l)));
}

// n / d: the hardware reciprocal (1 ulp) and one correction step
__device__ __forceinline__ float fast_rcp(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ D2 div(D2 n, D2 d) {
  const float r = fast_rcp(d.h);
  const float q = __fmul_rn(n.h, r);
  // n - q d, exact in the leading words
  float m = __fmaf_rn(-q, d.h, n.h);
  m = __fadd_rn(m, __fmaf_rn(-q, d.l, n.l));
  const float h = __fmaf_rn(m, r, q);  // renorm(q, m r)
  return D2{h, __fmaf_rn(m, r, -__fadd_rn(h, -q))};
}
// 1 / sqrt(x): the hardware approximation and one Newton step in pairs
__device__ __forceinline__ D2 rsqrt2(D2 x) {
  const float y = rsqrtf(x.h);
  const float p = __fmul_rn(y, y), e = __fmaf_rn(y, y, -p);
  const float a = __fmul_rn(x.h, p);
  float b = __fmaf_rn(x.h, p, -a);
  b = __fmaf_rn(x.h, e, b);
  b = __fmaf_rn(x.l, p, b);
  const float t = __fadd_rn(__fadd_rn(1.f, -a), -b);  // 1 - x y^2
  return renorm(y, __fmul_rn(__fmul_rn(0.5f, y), t));
}

// The range in which a double becomes a pair: below 2^-126 it is 0, from
// 2^kBigExp on (infinities and NaN included) NaN, which every later
// operation carries on, so that one test of a result tells whether all of
// its inputs were in range.
constexpr int kBigExp = 40;

// double -> pair by integer operations (the conversion instruction would
// take the FP64 pipe as long as an arithmetic one): h the leading 24 bits of
// the significand, l the remaining 29 rounded to 24.
__device__ __forceinline__ D2 to_pair(double x) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  const unsigned a = hi & 0x7fffffffu, sign = hi & 0x80000000u;
  constexpr unsigned tiny = (unsigned)(1023 - 126) << 20, big = (unsigned)(1023 + kBigExp) << 20;
  // exponent field of h: that of x minus 896
  const unsigned hb = (__funnelshift_l(lo, a, 3) - (896u << 23)) | sign;
  const float f = __fmul_rn(__uint2float_rn(lo & 0x1fffffffu), 0x1p-52f);
  const bool in = a - tiny < big - tiny;
  D2 r;
  r.h = __uint_as_float(in ? hb : (a < tiny ? 0u : 0x7fc00000u));
  r.l = in ? __fmul_rn(f, __uint_as_float(hb & 0xff800000u)) : 0.f;
  return r;
}

// float -> double by integer operations; denormals count as zero
__device__ __forceinline__ double to_double(float x) {
  const unsigned b = __float_as_uint(x), a = b & 0x7fffffffu;
  const bool z = a < 0x00800000u;
  const unsigned hi = z ? 0u : ((a >> 3) + (896u << 20));
  return __hiloint2double((int)(hi | (b & 0x80000000u)), z ? 0 : (int)(b << 29));
}
__device__ __forceinline__ double to_double(D2 a) { return to_double(a.h) + to_double(a.l); }

// The same operations on doubles, for code written for either; as above
// without contraction, so that two uses of the same code give the same bits.
__device__ __forceinline__ double neg(double a) { return -a; }
__device__ __forceinline__ double add(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ double sub(double a, double b) { return __dadd_rn(a, -b); }
__device__ __forceinline__ double mul(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ double madd(double a, double b, double c) { return __fma_rn(a, b, c); }
__device__ __forceinline__ double square(double a) { return __dmul_rn(a, a); }
__device__ __forceinline__ double scale(double a, double p2) { return __dmul_rn(a, p2); }

// c ? -a : a
__device__ __forceinline__ D2 flip(bool c, D2 a) { return c ? neg(a) : a; }
__device__ __forceinline__ double flip(bool c, double a) { return c ? -a : a; }
// a b + c for a power of two a
__device__ __forceinline__ D2 scale_add(D2 b, float a, D2 c) { return add(scale(b, a), c); }
__device__ __forceinline__ double scale_add(double b, double a, double c) {
  return __fma_rn(b, a, c);
}

// a b - c d and a - b c (in FP64 without the rounding of one product)
template <class X>
__device__ __forceinline__ X mul_sub(X a, X b, X c, X d) { return sub(mul(a, b), mul(c, d)); }
template <class X>
__device__ __forceinline__ X sub_mul(X a, X b, X c) { return sub(a, mul(b, c)); }
__device__ __forceinline__ double mul_sub(double a, double b, double c, double d) {
  return madd(a, b, -mul(c, d));
}
__device__ __forceinline__ double sub_mul(double a, double b, double c) { return madd(-b, c, a); }

// c ? a : b, word by word
__device__ __forceinline__ D2 pick2(bool c, D2 a, D2 b) {
  return D2{c ? a.h : b.h, c ? a.l : b.l};
}
__device__ __forceinline__ double pick2(bool c, double a, double b) { return c ? a : b; }

// Two pairs in the lanes of packed FP32 instructions (fma / add / mul .f32x2,
// which take 2 cycles for both lanes, negated operands included): half the
// instructions to issue and to fetch. Each lane rounds as the scalar form.
struct Q2 {
  float2 h, l;
};
__device__ __forceinline__ float2 neg2(float2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ float2 dup(float a) { return make_float2(a, a); }
__device__ __forceinline__ Q2 both(D2 a, D2 b) {
  return Q2{make_float2(a.h, b.h), make_float2(a.l, b.l)};
}
__device__ __forceinline__ Q2 both(D2 a) { return both(a, a); }
__device__ __forceinline__ D2 first(Q2 a) { return D2{a.h.x, a.l.x}; }
__device__ __forceinline__ D2 second(Q2 a) { return D2{a.h.y, a.l.y}; }
__device__ __forceinline__ Q2 renorm(float2 s, float2 e) {
  const float2 h = __fadd2_rn(s, e);
  return Q2{h, __fadd2_rn(e, neg2(__fadd2_rn(h, neg2(s))))};
}
__device__ __forceinline__ Q2 neg(Q2 a) { return Q2{neg2(a.h), neg2(a.l)}; }
__device__ __forceinline__ Q2 add(Q2 a, Q2 b) {
  const float2 s = __fadd2_rn(a.h, b.h);
  const float2 t = __fadd2_rn(s, neg2(a.h));
  const float2 e = __fadd2_rn(__fadd2_rn(a.h, neg2(__fadd2_rn(s, neg2(t)))),
                              __fadd2_rn(b.h, neg2(t)));
  return renorm(s, __fadd2_rn(e, __fadd2_rn(a.l, b.l)));
}
__device__ __forceinline__ Q2 sub(Q2 a, Q2 b) { return add(a, neg(b)); }
__device__ __forceinline__ Q2 mul(Q2 a, Q2 b) {
  const float2 p = __fmul2_rn(a.h, b.h);
  float2 e = __ffma2_rn(a.h, b.h, neg2(p));
  e = __ffma2_rn(a.h, b.l, e);
  e = __ffma2_rn(a.l, b.h, e);
  return renorm(p, e);
}
__device__ __forceinline__ Q2 mul(Q2 a, float c) {
  const float2 p = __fmul2_rn(a.h, dup(c));
  return renorm(p, __ffma2_rn(a.l, dup(c), __ffma2_rn(a.h, dup(c), neg2(p))));
}
__device__ __forceinline__ Q2 square(Q2 a) {
  const float2 p = __fmul2_rn(a.h, a.h);
  return renorm(p, __ffma2_rn(__fadd2_rn(a.h, a.h), a.l, __ffma2_rn(a.h, a.h, neg2(p))));
}
__device__ __forceinline__ Q2 scale(Q2 a, float2 p2) {
  return Q2{__fmul2_rn(a.h, p2), __fmul2_rn(a.l, p2)};
}
__device__ __forceinline__ Q2 scale(Q2 a, float p2) { return scale(a, dup(p2)); }
__device__ __forceinline__ Q2 scale_add(Q2 b, float a, Q2 c) { return add(scale(b, a), c); }
__device__ __forceinline__ Q2 abs2(Q2 a) { return both(abs2(first(a)), abs2(second(a))); }
__device__ __forceinline__ Q2 madd(Q2 a, Q2 b, Q2 c) {
  const float2 p = __fmul2_rn(a.h, b.h);
  float2 e = __ffma2_rn(a.h, b.h, neg2(p));
  e = __ffma2_rn(a.h, b.l, e);
  e = __ffma2_rn(a.l, b.h, e);
  const float2 s = __fadd2_rn(p, c.h);
  const float2 t = __fadd2_rn(s, neg2(p));
  const float2 r = __fadd2_rn(__fadd2_rn(p, neg2(__fadd2_rn(s, neg2(t)))),
                              __fadd2_rn(c.h, neg2(t)));
  return renorm(s, __fadd2_rn(r, __fadd2_rn(e, c.l)));
}
__device__ __forceinline__ Q2 div(Q2 n, Q2 d) {
  const float2 r = make_float2(fast_rcp(d.h.x), fast_rcp(d.h.y));
  const float2 q = __fmul2_rn(n.h, r);
  float2 m = __ffma2_rn(neg2(q), d.h, n.h);
  m = __fadd2_rn(m, __ffma2_rn(neg2(q), d.l, n.l));
  const float2 h = __ffma2_rn(m, r, q);
  return Q2{h, __ffma2_rn(m, r, neg2(__fadd2_rn(h, neg2(q))))};
}

__device__ __forceinline__ Q2 pick2(bool c, Q2 a, Q2 b) {
  return both(pick2(c, first(a), first(b)), pick2(c, second(a), second(b)));
}

// What generic code needs to know of a number type X (D2 or double).
template <class X>
struct Num;
template <>
struct Num<D2> {
  using Scale = float;  // leading word, and type of a power of two
  static __device__ __forceinline__ constexpr D2 c(double x) { return dconst(x); }
  static __device__ __forceinline__ float lead(D2 x) { return x.h; }
  // 2^e and 2^-e of the exponent e of x > 0 (2^e <= x)
  static __device__ __forceinline__ void exponent(float x, float& up, float& down) {
    const unsigned e = __float_as_uint(x) & 0x7f800000u;
    up = __uint_as_float(e);
    down = __uint_as_float((254u << 23) - e);
  }
};
template <>
struct Num<Q2> {
  using Scale = float;
  static __device__ __forceinline__ Q2 c(double x) { return both(dconst(x)); }
};
template <>
struct Num<double> {
  using Scale = double;
  static __device__ __forceinline__ constexpr double c(double x) { return x; }
};

}  // namespace hweno
