// The nonlinear part of the L-HWENO reconstruction and limiter (Zhang & Zhao,
// arXiv:2207.05258, Sec. 2.1-2.2) for FP64 states in pairs of FP32 numbers
// (dfloat.cuh).
//
// The scheme splits exactly into a linear part, taken in FP64 or relative to
// an FP64 value, and a correction. With w_l = g_l (1 + tau / b_l) / S and
// b_l = beta_l + eps the nonlinear value is
//   sum of the paper's combination = p_0 + C,
//   C = phi_1 (p_1 - p_0) + phi_2 (p_2 - p_0),
//   phi_1 = tau g_1 b_2 (b_0 - b_1) / D, phi_2 = tau g_2 b_1 (b_0 - b_2) / D,
//   D = b_0 b_1 b_2 + tau (g_0 b_1 b_2 + g_1 b_0 b_2 + g_2 b_0 b_1),
// up to the common factor that the free choice of p_0's share leaves, and
// p_0 commutes with the characteristic projection. So only C needs the
// projection, and it depends on differences of the data alone.
//
// A pair carries 48 bits: C has an error of about 2^-46 (phi_1 |p_1 - p_0| +
// phi_2 |p_2 - p_0|), and where the linear part is taken in pairs that has one
// of 2^-48 of the differences. The FP64 form starts from the full values and
// has an error of a few 2^-53 of alpha U. Items are evaluated in pairs while
// their error stays below that: kWeakPhi, kWeakLevel and the like here,
// interface_route in line_df.cuh. Where they fail (shocks, under-resolved jumps
// and waves, noise, and whatever leaves the FP32 range: any overflow or NaN
// fails the same tests) the caller evaluates the item in FP64.
#pragma once

#include <type_traits>

#include "dfloat.cuh"

namespace hweno {

// Leading 24 bits (truncated) of a double as a float by integer operations;
// NaN outside the float range, 0 below it.
__device__ __forceinline__ float to_float(double x) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  const unsigned a = hi & 0x7fffffffu;
  constexpr unsigned tiny = (unsigned)(1023 - 126) << 20, big = (unsigned)(1023 + 127) << 20;
  const unsigned hb = (__funnelshift_l(lo, a, 3) - (896u << 23)) | (hi & 0x80000000u);
  return __uint_as_float(a - tiny < big - tiny ? hb : (a < tiny ? 0u : 0x7fc00000u));
}

// 1 / x for a double: the FP32 reciprocal (23 bits) and one step of the
// third-order Newton (Householder) iteration, y (1 + e + e^2) with
// e = 1 - x y: three FP64 operations, about one unit in the last place. The
// division where x lies outside the range of to_float or 1 / x might.
__device__ __forceinline__ double recip_fp64(double x) {
  const float f = to_float(x);
  if (!(fabsf(f) >= 0x1p-100f && fabsf(f) <= 0x1p100f)) return 1.0 / x;
  const double y = to_double(fast_rcp(f));
  const double e = __fma_rn(-x, y, 1.0);
  return __fma_rn(y, __fma_rn(e, e, e), y);
}

// 1 / sqrt(x) in the same way, y (1 + e / 2 + 3 e^2 / 8) with e = 1 - x y^2:
// five FP64 operations.
__device__ __forceinline__ double rsqrt_fp64(double x) {
  const float f = to_float(x);
  if (!(f >= 0x1p-100f && f <= 0x1p100f)) return rsqrt(x);
  const double y = to_double(rsqrtf(f));
  const double e = __fma_rn(-__dmul_rn(x, y), y, 1.0);
  return __fma_rn(__dmul_rn(y, e), __fma_rn(0.375, e, 0.5), y);
}

// Weights of the reconstruction or the limiter, eps, and the largest beta
// for which the products of pairs stay in range.
template <class X>
struct LineWeights {
  X g0, g1, g2, eps;
  float bmax;
};

// An item is weak while every phi is at most kWeakPhi or the sum of phi
// |differences| over the sides and fields that exceed it is at most a fraction
// of the local alpha U: kWeakLevel (Euler interfaces), kWeakScalar (interfaces
// of the scalar equations, whose differences may be as large as their values),
// kWeakLimiter of U (limiter on characteristic fields; on components, whose
// FP64 form starts from differences, the first test alone). Error of L^1, L^2
// and v~ over the FP64 form's (2-norms, waves of 5 to 800 points, noise of
// 1e-8 to 0.3, jumps, steep profiles; tests/test_host_pairs.py): at most 1.
// With kWeakPhi = 1/32, one level of 1/64 for all and no bound on the
// differences it reached 26 (noise about zero), 8 (waves of 7 points) and 24
// (v~ of a wave of 15 points). On flows as they are run (Riemann problems, blast,
// Burgers and density waves, Mach 2, 1 to 20 steps, against 128 bits): U 0.5-1.1,
// V, W 0.2-0.85, L^1 0.1-0.5, L^2, L^3 0.04-0.84, v~ 0.01-0.6.
constexpr float kWeakPhi = 1.f / 256.f, kWeakLevel = 1.f / 64.f, kWeakScalar = 1.f / 1024.f,
                kWeakLimiter = 1.f / 4096.f;

// The smoothness indicators b_l of one side of an interface from the
// differences of its stencil: y1 = f_{i-1} - f_i + H_i,
// y2 = f_i - f_{i+1} + H_i, s = H_{i-1} + H_{i+1} - 2 H_i,
// d = H_{i-1} - H_{i+1} and H_i. beta_0 as the sum of squares of the
// quadratic form's triangular factorisation (its odd part in H_i, s,
// g = y1 + y2, its even part in d, lap = y1 - y2); the square of H_i is
// common to the three.
template <class X>
__device__ __forceinline__ void flux_indicators(X y1, X y2, X s, X d, X H0, X g, X lap, X eps,
                                                X& b0, X& b1, X& b2) {
  using N = Num<X>;
  const X z1 = madd(N::c(9883630.0 / 3288933.0), g, s);
  const X z2 = madd(N::c(44358.0 / 22025.0), lap, d);
  const X h = add(square(H0), eps);
  b0 = madd(N::c(1096311.0 / 1120.0), square(z1), h);
  b0 = madd(N::c(21520059541.0 / 2210162976.0), square(g), b0);
  b0 = madd(N::c(4405.0 / 112.0), square(z2), b0);
  b0 = madd(N::c(1421461.0 / 1321500.0), square(lap), b0);
  b1 = madd(N::c(13.0 / 3.0), square(y1), h);
  b2 = madd(N::c(13.0 / 3.0), square(y2), h);
}
// The limiter's from q1 = u_i - u_{i-1}, q2 = u_{i+1} - u_i, lap = q2 - q1,
// du = q1 + q2, dV = Vm - Vp and r = Vm + Vp - du (Vm, Vp = dx v_{i-1},
// dx v_{i+1}).
template <class X>
__device__ __forceinline__ void limiter_indicators(X q1, X q2, X lap, X du, X dV, X r, X eps,
                                                   X& b0, X& b1, X& b2) {
  using N = Num<X>;
  const X z1 = madd(N::c(-120.0 / 3169.0), du, r);
  const X z2 = madd(N::c(527690.0 / 262907.0), lap, dV);
  b0 = madd(N::c(3169.0 / 1280.0), square(z1), eps);
  b0 = madd(N::c(781.0 / 3169.0), square(du), b0);
  b0 = madd(N::c(262907.0 / 6720.0), square(z2), b0);
  b0 = madd(N::c(1421461.0 / 1314535.0), square(lap), b0);
  b1 = add(square(q1), eps);
  b2 = add(square(q2), eps);
}

// A word of a pair and of two packed pairs: what correction() does lane by
// lane.
__device__ __forceinline__ void to_unit(float mx, float& up, float& down) {
  Num<D2>::exponent(mx, up, down);
}
__device__ __forceinline__ void to_unit(float2 mx, float2& up, float2& down) {
  to_unit(mx.x, up.x, down.x);
  to_unit(mx.y, up.y, down.y);
}
__device__ __forceinline__ float max3(float a, float b, float c) { return fmaxf(a, fmaxf(b, c)); }
__device__ __forceinline__ float2 max3(float2 a, float2 b, float2 c) {
  return make_float2(max3(a.x, b.x, c.x), max3(a.y, b.y, c.y));
}
__device__ __forceinline__ float quarter(float a) { return 0.25f * a; }
__device__ __forceinline__ float2 quarter(float2 a) { return __fmul2_rn(a, dup(0.25f)); }
// Adds to e a bound of phi (|p| + |q|) where phi exceeds kWeakPhi, phi taken
// with b_0 for b_0 - b_l: what the difference's own error is a fraction of.
__device__ __forceinline__ void bound(float& e, float tau, float q1, float q2, float b0, float den,
                                      float p, float q, float mx, float bmax) {
  const float top = tau * (fmaxf(q1, q2) * b0);
  if (!(top <= kWeakPhi * den)) e += top * fast_rcp(den) * (fabsf(p) + fabsf(q));
  if (!(mx < bmax)) e = __int_as_float(0x7f800000);
}
__device__ __forceinline__ void bound(float2& e, float2 tau, float2 q1, float2 q2, float2 b0,
                                      float2 den, float2 p, float2 q, float2 mx, float bmax) {
  bound(e.x, tau.x, q1.x, q2.x, b0.x, den.x, p.x, q.x, mx.x, bmax);
  bound(e.y, tau.y, q1.y, q2.y, b0.y, den.y, p.y, q.y, mx.y, bmax);
}

// (phi_1 - phi_2) p + (phi_1 + phi_2) q from b_l in pairs; where a phi_l
// exceeds kWeakPhi, adds a bound of phi (|p| + |q|) to e (infinite or NaN
// where the arithmetic has left its range). X: D2, or Q2 with e per lane.
template <class X, class E>
__device__ __forceinline__ X correction(X b0, X b1, X b2, X p, X q, const LineWeights<X>& w, E& e) {
  // the indicators scaled by a power of two to at most 2 (products of three
  // of them and tau stay in range); tau = t^2 / 4 scales back by that power
  const E mx = max3(b0.h, b1.h, b2.h);
  E up, down;
  to_unit(mx, up, down);
  b0 = scale(b0, down);
  b1 = scale(b1, down);
  b2 = scale(b2, down);
  const X e1 = sub(b0, b1), e2 = sub(b0, b2);
  const X tau = scale(square(add(abs2(e1), abs2(e2))), quarter(up));
  const X q1 = mul(w.g1, b2), q2 = mul(w.g2, b1);
  const X n1 = mul(q1, e1), n2 = mul(q2, e2);
  const X den = madd(mul(b1, b2), madd(w.g0, tau, b0), mul(mul(tau, b0), add(q1, q2)));
  const X num = mul(tau, madd(p, sub(n1, n2), mul(q, add(n1, n2))));
  bound(e, tau.h, q1.h, q2.h, b0.h, den.h, p.h, q.h, mx, w.bmax);
  return div(num, den);
}

// 12 C of one side of an interface (Q2: of both): 60 (p_1 - p_0) = 5 g - 3 m
// and 60 (p_2 - p_0) = -5 g - 3 m with m = d + 2 lap.
template <class X, class E>
__device__ __forceinline__ X side_correction(X y1, X y2, X s, X d, X H0, const LineWeights<X>& w,
                                             E& e) {
  const X g = add(y1, y2), lap = sub(y1, y2);
  X b0, b1, b2;
  flux_indicators(y1, y2, s, d, H0, g, lap, w.eps, b0, b1, b2);
  const X m = mul(add(d, scale(lap, 2.f)), Num<X>::c(-3.0 / 5.0));
  return correction(b0, b1, b2, g, m, w, e);
}

// 4 times the correction of dx v~_i to the linear dx q_0':
// 4 (q_1 - q_0) = r - 2 lap, 4 (q_2 - q_0) = r + 2 lap.
template <class X, class E>
__device__ __forceinline__ X limiter_correction(X q1, X q2, X Vm, X Vp, const LineWeights<X>& w,
                                                E& e) {
  const X lap = sub(q2, q1), du = add(q1, q2), dV = sub(Vm, Vp), r = sub(add(Vm, Vp), du);
  X b0, b1, b2;
  limiter_indicators(q1, q2, lap, du, dV, r, w.eps, b0, b1, b2);
  return correction(b0, b1, b2, scale(lap, -2.f), r, w, e);
}

// In FP64 the value itself in the form of the paper's weights,
// (W_0 (p_0 - g_1 p_1 - g_2 p_2) + W_1 p_1 + W_2 p_2) / (g_0 W_0 + W_1 + W_2)
// with W_l of the size of (b_l + tau) prod_{m != l} b_m: beside a jump the
// weights discard candidates far larger than the result, which a linear part
// and a correction that cancels it would not resolve.
__device__ __forceinline__ double weighted(double b0, double b1, double b2, double p0, double p1,
                                           double p2, const LineWeights<double>& w) {
  // scaled to at most 2 by their exponent fields (the largest is the
  // maximum of non-negative bit patterns)
  const int top = max(__double2hiint(b0), max(__double2hiint(b1), __double2hiint(b2)));
  const int e = top & 0x7ff00000;
  const double up = __hiloint2double(e, 0);
  auto shift = [&](double x) {  // x 2^-exponent; 0 below the normal range
    const int h = __double2hiint(x) - (e - (1023 << 20));
    return h >= (1 << 20) ? __hiloint2double(h, __double2loint(x)) : 0.0;
  };
  if (e != 0x7ff00000) {  // (an infinity or NaN stays and shows in the result)
    b0 = shift(b0);
    b1 = shift(b1);
    b2 = shift(b2);
  }
  const double t = add(fabs(sub(b0, b1)), fabs(sub(b0, b2)));
  const double tau = mul(mul(mul(0.25, t), t), up);
  const double P12 = mul(b1, b2), P = mul(b0, P12), tb = mul(tau, b0);
  const double W0 = madd(tau, P12, P);
  const double W1 = mul(w.g1, madd(tb, b2, P)), W2 = mul(w.g2, madd(tb, b1, P));
  // the small products first, so that one operation each rounds the full sums
  const double r = sub(p0, madd(w.g2, p2, mul(w.g1, p1)));
  const double num = madd(W0, r, madd(W1, p1, mul(W2, p2)));
  const double den = madd(w.g0, W0, add(W1, W2)), id = recip_fp64(den), q = mul(num, id);
  return madd(madd(-q, den, num), id, q);
}
// f-hat of a side minus the side's split flux at its own point:
// 6 (p_1 - f_i) = y1 + 3 H_i, 6 (p_2 - f_i) = 3 H_i - y2,
// 60 (p_0 - f_i) = 11 lap + 3 d + 30 H_i.
__device__ __forceinline__ double side_value(double y1, double y2, double s, double d, double H0,
                                             const LineWeights<double>& w) {
  const double g = add(y1, y2), lap = sub(y1, y2), h3 = mul(0.5, H0);
  double b0, b1, b2;
  flux_indicators(y1, y2, s, d, H0, g, lap, w.eps, b0, b1, b2);
  return weighted(b0, b1, b2, madd(11.0 / 60.0, lap, madd(0.05, d, h3)), madd(1.0 / 6.0, y1, h3),
                  madd(-1.0 / 6.0, y2, h3), w);
}
// dx v~_i
__device__ __forceinline__ double limiter_value(double q1, double q2, double Vm, double Vp,
                                                const LineWeights<double>& w) {
  const double lap = sub(q2, q1), du = add(q1, q2), dV = sub(Vm, Vp), sV = add(Vm, Vp);
  const double r = sub(sV, du);
  double b0, b1, b2;
  limiter_indicators(q1, q2, lap, du, dV, r, w.eps, b0, b1, b2);
  return weighted(b0, b1, b2, madd(0.75, du, mul(-0.25, sV)), q1, q2, w);
}

// Characteristic system of the Euler flux Jacobian in direction DIR (M = 3:
// 1D, M = 4: 2D) in the factored form of Char1 / Char2: fields 0, 1, 2 belong
// to u - c, u, u + c, field 3 (2D) to the shear wave. Component slots:
// density 0, normal momentum kn, tangential kt, energy M - 1.
template <class X, int M, int DIR>
struct LineChar {
  static constexpr int kn = 1 + DIR, kt = 2 - DIR, kE = M - 1;
  X un, ut, H, c, q, b, bq, bu, bt, hic, huc;
  LineChar() = default;
  __device__ __forceinline__ void init(X un_, X ut_, X H_, X q_, X c2, X gm1) {
    un = un_;
    ut = ut_;
    H = H_;
    q = q_;
    X ic;
    if constexpr (std::is_same<X, double>::value) ic = rsqrt_fp64(c2);
    else ic = rsqrt2(c2);
    c = mul(c2, ic);
    b = scale(mul(gm1, square(ic)), 0.5f);
    bq = mul(b, q);
    bu = mul(b, un);
    if constexpr (M == 4) bt = mul(b, ut);
    hic = scale(ic, 0.5f);
    huc = mul(hic, un);
  }
  // what factors() needs, in both lanes
  __device__ __forceinline__ LineChar<Q2, M, DIR> packed() const {
    LineChar<Q2, M, DIR> r;
    if constexpr (std::is_same<X, D2>::value) {
      r.b = both(b);
      r.bq = both(bq);
      r.bu = both(bu);
      r.hic = both(hic);
      r.huc = both(huc);
      if constexpr (M == 4) {
        r.bt = both(bt);
        r.ut = both(ut);
      }
    }
    return r;
  }
  // a field's bound in units of the density (the shear field is a momentum)
  __device__ __forceinline__ float density_units(int q, float e) const {
    if constexpr (M == 4 && std::is_same<X, D2>::value)
      return q == 3 ? e * fast_rcp(c.h) : e;
    else
      return e;
  }
  // kinetic energy per mass
  static __device__ __forceinline__ X kinetic(X un, X ut) {
    X s = square(un);
    if constexpr (M == 4) s = madd(ut, ut, s);
    return scale(s, 0.5f);
  }
  // The factors of L x: its fields are A + B, x_0 - 2 A, A - B and S.
  struct Factors {
    X x0, A, B, S;
    // field q of L x (a run-time q, so that loops over the fields need no
    // unrolling)
    __device__ __forceinline__ X field(int q) const {
      using P2 = typename Num<X>::Scale;
      const X p = pick2(q == 1, x0, A), r = pick2(q == 1, A, B);
      const X v = scale_add(r, q == 0 ? P2(1) : q == 1 ? P2(-2) : P2(-1), p);
      if constexpr (M == 4) return pick2(q == 3, S, v);
      else return v;
    }
  };
  __device__ __forceinline__ Factors factors(const X* x) const {
    Factors f;
    f.x0 = x[0];
    f.A = madd(b, x[kE], mul_sub(bq, x[0], bu, x[kn]));
    if constexpr (M == 4) f.A = sub_mul(f.A, bt, x[kt]);
    f.B = mul_sub(huc, x[0], hic, x[kn]);
    if constexpr (M == 4) f.S = sub_mul(x[kt], ut, x[0]);
    return f;
  }
  // R s
  __device__ __forceinline__ void right(const X* s, X* out) const {
    const X s02 = add(s[0], s[2]), sum = add(s02, s[1]), dif = mul(c, sub(s[2], s[0]));
    out[0] = sum;
    out[kn] = madd(un, sum, dif);
    X e = madd(H, s02, madd(q, s[1], mul(un, dif)));
    if constexpr (M == 4) {
      out[kt] = madd(ut, sum, s[3]);
      e = madd(ut, s[3], e);
    }
    out[kE] = e;
  }
};

// 60 times an interface's linear part relative to (F_i + F_{i+1}) / 2, one
// component: the sum of 11 y1 + 19 y2 + 3 d over the two sides.
template <class X>
__device__ __forceinline__ X linear_part(X y1, X y2, X d) {
  return add(mul(y1, 11.f), add(mul(y2, 19.f), mul(d, 3.f)));
}

// 4 times one side's dx p_0' (Sec. 2.1, the derivative flux), one component;
// the "-" side's with its reversed and negated rows is minus its share.
template <class X>
__device__ __forceinline__ X derivative_part(X y1, X y2, X s, X d, X H0) {
  return add(scale(H0, 4.f), add(add(y1, d), madd(Num<X>::c(-2.0 / 3.0), s, mul(y2, -7.f))));
}

// Maximum over the warp of non-negative doubles (their bits order as
// unsigned integers), by integer reductions: a double maximum costs FP64
// compares. The result is valid in every lane.
__device__ __forceinline__ unsigned long long warp_max_bits(double v) {
  const unsigned hi = (unsigned)__double2hiint(v), lo = (unsigned)__double2loint(v);
  const unsigned mh = __reduce_max_sync(0xffffffffu, hi);
  const unsigned ml = __reduce_max_sync(0xffffffffu, hi == mh ? lo : 0u);
  return ((unsigned long long)mh << 32) | ml;
}

}  // namespace hweno
