// One line direction of the L-HWENO stage for FP64 states (Zhang & Zhao,
// arXiv:2207.05258, Sec. 2.1-2.2), shared by the 1D and 2D stage kernels:
// the data of a tile's points in shared memory and the evaluation of
// interface fluxes and limited derivatives along the line, in pairs of FP32
// numbers where the correction is small (weno_df.cuh) and in FP64 elsewhere.
#pragma once

#include <type_traits>

#include "hweno.h"
#include "hweno_math.cuh"
#include "internal.h"
#include "weno_df.cuh"

#ifndef HWENO_UNROLL_FIELDS
#define HWENO_UNROLL_FIELDS 1
#endif

namespace hweno {

constexpr int kUnrollFields = HWENO_UNROLL_FIELDS;

// Shared memory of a tile of L loaded points (flat index k; the neighbours
// of k along the line are k - S and k + S) and LI interfaces or updated
// points. M components, direction DIR, MX extra double rows for the caller.
// Rows of doubles: U, N (the derivative along the line), F, h = A N (Euler:
// M - 1 rows, F_0 = U_kn and h_0 = N_kn), extras. Rows of pairs: H^+, H^-
// and dx N (points), P = (dF + alpha dU)/2, M = (dF - alpha dU)/2 and dU
// (edges k, k + S), and for Euler sqrt(rho), un, H and (2D) ut. Then
// the outputs: c = f-hat - (F_i + F_{i+1})/2, the derivative flux D, and the
// limited derivative.
template <int M_, int DIR, bool EUL_, int MX = 0, bool SLIM_ = false>
struct LineTile {
  static constexpr int M = M_, kn = EUL_ ? 1 + DIR : 0;
  static constexpr bool EUL = EUL_, SLIM = SLIM_;
  static constexpr int NE = EUL ? M : 0;
  static constexpr int MF = EUL ? M - 1 : M;  // stored rows of F and h
  static constexpr int nd = 2 * M + 2 * MF + MX, np = (SLIM ? 4 : 6) * M + NE, no = 3 * M;
  __host__ __device__ static constexpr size_t bytes(int L, int LI) {
    return sizeof(double) * ((size_t)(nd + np) * L + (size_t)no * LI);
  }
  double* base;
  int L, LI;
  unsigned* st;  // checked builds: every row and column is checked
  D2 ial;        // SLIM: 1 / alpha
  __device__ __forceinline__ int at(int row, int rows, int k, int len) const {
#if defined(HWENO_CHECKS) && HWENO_CHECKS
    if ((unsigned)row >= (unsigned)rows || (unsigned)k >= (unsigned)len) {
      atomicOr(st, STATUS_BOUNDS);
      return 0;
    }
#endif
    return row * len + k;
  }
  __device__ __forceinline__ double& d(int row, int k) const { return base[at(row, nd, k, L)]; }
  __device__ __forceinline__ D2& p(int row, int k) const {
    return reinterpret_cast<D2*>(base + nd * L)[at(row, np, k, L)];
  }
  // a pair row as doubles (double_rows)
  __device__ __forceinline__ double& pd(int row, int k) const {
    return base[nd * L + at(row, np, k, L)];
  }
  __device__ __forceinline__ double& o(int row, int j) const {
    return base[(nd + np) * L + at(row, no, j, LI)];
  }
  __device__ __forceinline__ double& U(int c, int k) const { return d(c, k); }
  __device__ __forceinline__ double& N(int c, int k) const { return d(M + c, k); }
  __device__ __forceinline__ double& F(int c, int k) const {
    if constexpr (EUL) return c == 0 ? d(kn, k) : d(2 * M + c - 1, k);
    else return d(2 * M + c, k);
  }
  __device__ __forceinline__ double& h(int c, int k) const {
    if constexpr (EUL) return c == 0 ? d(M + kn, k) : d(2 * M + MF + c - 1, k);
    else return d(2 * M + MF + c, k);
  }
  __device__ __forceinline__ double& extra(int r, int k) const { return d(2 * M + 2 * MF + r, k); }
  // split pairs of side sd (0: H^+, P; 1: -H^-, -M)
  __device__ __forceinline__ D2& H(int sd, int c, int k) const { return p(sd * M + c, k); }
  __device__ __forceinline__ D2& X(int sd, int c, int k) const { return p((2 + sd) * M + c, k); }
  __device__ __forceinline__ D2 dU(int c, int k) const {
    if constexpr (SLIM) return mul(add(X(0, c, k), X(1, c, k)), ial);
    else return p(4 * M + c, k);
  }
  __device__ __forceinline__ float dU_lead(int c, int k) const {
    if constexpr (SLIM) return (X(0, c, k).h + X(1, c, k).h) * ial.h;
    else return p(4 * M + c, k).h;
  }
  __device__ __forceinline__ D2 Nx(int c, int k) const {
    if constexpr (SLIM) return mul(add(H(0, c, k), H(1, c, k)), ial);
    else return p(5 * M + c, k);
  }
  // eigen-system inputs: sqrt(rho), un, H, ut
  __device__ __forceinline__ D2& E(int e, int k) const { return p((SLIM ? 4 : 6) * M + e, k); }
  __device__ __forceinline__ double& C(int c, int j) const { return o(c, j); }
  __device__ __forceinline__ double& D(int c, int j) const { return o(M + c, j); }
  __device__ __forceinline__ double& lim(int c, int j) const { return o(2 * M + c, j); }
};

// Weights of the reconstruction (lim = false) or the limiter as X.
template <class X>
__device__ __forceinline__ LineWeights<X> line_weights(const SchemeParams& sp, bool lim) {
  const int o = lim ? 3 : 0;
  if constexpr (std::is_same<X, double>::value)
    return LineWeights<double>{sp.wd[o], sp.wd[o + 1], sp.wd[o + 2], sp.wd[6], 0.f};
  else
    return LineWeights<D2>{sp.wp[o], sp.wp[o + 1], sp.wp[o + 2], sp.wp[6], sp.wp_bmax};
}
__device__ __forceinline__ D2 gm1_pair(const SchemeParams& sp) { return sp.wp[7]; }

// A pair of a quantity that sets the scale of the data (density, wave
// speed): NaN below 2^-30, where differences of tiny data could fall under
// the pairs' range; what depends on it is then evaluated in FP64.
__device__ __forceinline__ D2 scale_pair(double x) {
  D2 r = to_pair(x);
  if (!(r.h >= 0x1p-30f)) r.h = __int_as_float(0x7fc00000);
  return r;
}

// The pairs of point k, component c, from the derivative N and h = A N of its
// state: H^{+-} = dx (h +- alpha N) / 2 and dx N.
template <class T>
__device__ __forceinline__ void point_pair(const T& r, int c, int k, double N, double h, D2 alp,
                                           D2 dxp) {
  const D2 nx = mul(dxp, to_pair(N)), x = mul(dxp, to_pair(h)), y = mul(alp, nx);
  if constexpr (!T::SLIM) r.p(5 * T::M + c, k) = nx;
  r.H(0, c, k) = scale(add(x, y), 0.5f);
  r.H(1, c, k) = scale(sub(y, x), 0.5f);
}
template <class T>
__device__ __forceinline__ void point_pairs(const T& r, int k, const double* N, const double* h,
                                            D2 alp, D2 dxp) {
#pragma unroll
  for (int c = 0; c < T::M; ++c) point_pair(r, c, k, N[c], h[c], alp, dxp);
}

// The eigen-system's inputs at point k from rho, 1/rho, E + p and the
// velocities along and across the line.
template <class T>
__device__ __forceinline__ void point_eigen(const T& r, int k, double rho, double ir, double Ep,
                                            double un, double ut) {
  const D2 rp = scale_pair(rho);
  r.E(0, k) = mul(rp, rsqrt2(rp));
  r.E(1, k) = to_pair(un);
  r.E(2, k) = mul(to_pair(Ep), to_pair(ir));
  if constexpr (T::M == 4) r.E(3, k) = to_pair(ut);
}

// Component c of the edge between points k and k + S.
template <class T>
__device__ __forceinline__ void edge_pair(const T& r, int c, int k, int S, D2 alp) {
  const D2 dU = to_pair(sub(r.U(c, k + S), r.U(c, k)));
  const D2 dF = to_pair(sub(r.F(c, k + S), r.F(c, k))), au = mul(alp, dU);
  if constexpr (!T::SLIM) r.p(4 * T::M + c, k) = dU;
  r.X(0, c, k) = scale(add(dF, au), 0.5f);
  r.X(1, c, k) = scale(sub(au, dF), 0.5f);
}
template <class T>
__device__ __forceinline__ void edge_pairs(const T& r, int k, int S, D2 alp) {
  D2 dU[T::M];
#pragma unroll
  for (int c = 0; c < T::M; ++c) {
    dU[c] = to_pair(sub(r.U(c, k + S), r.U(c, k)));
    if constexpr (!T::SLIM) r.p(4 * T::M + c, k) = dU[c];
  }
#pragma unroll
  for (int c = 0; c < T::M; ++c) {
    const D2 dF = T::EUL && c == 0 ? dU[T::kn] : to_pair(sub(r.F(c, k + S), r.F(c, k)));
    const D2 au = mul(alp, dU[c]);
    r.X(0, c, k) = scale(add(dF, au), 0.5f);
    r.X(1, c, k) = scale(sub(au, dF), 0.5f);
  }
}

// The data of a line as X: pairs from the tile's pair rows, or doubles
// formed from its double rows (ROWS: where they are of more than one double,
// read from the rows that double_rows has made of them).
template <class X, class T, bool ROWS = false>
struct LineData;
template <class T>
struct LineData<D2, T, false> {
  const T& r;
  int S;
  const SchemeParams& sp;
  __device__ __forceinline__ LineData(const T& r_, int S_, double, double, const SchemeParams& sp_)
      : r(r_), S(S_), sp(sp_) {}
  __device__ __forceinline__ D2 H(int sd, int c, int k) const { return r.H(sd, c, k); }
  __device__ __forceinline__ D2 X(int sd, int c, int k) const { return r.X(sd, c, k); }
  __device__ __forceinline__ D2 dU(int c, int k) const { return r.dU(c, k); }
  __device__ __forceinline__ D2 Nx(int c, int k) const { return r.Nx(c, k); }
  __device__ __forceinline__ D2 gm1() const { return gm1_pair(sp); }
  // velocities and enthalpy at point k, or of the Roe average or the mean state
  // of k and k + S
  __device__ __forceinline__ void state(int k, bool edge, D2& un, D2& ut, D2& H) const {
    if (!edge) {
      un = r.E(1, k);
      H = r.E(2, k);
      if constexpr (T::M == 4) ut = r.E(3, k);
      return;
    }
    const D2 sl = r.E(0, k), sr = r.E(0, k + S);
    if (sp.eig_avg != 0) {  // mean state (gamma E = rho H + (gamma - 1) rho q)
      const D2 rl = square(sl), rr = square(sr), ir = div(D2{1.f, 0.f}, add(rl, rr));
      auto mean = [&](D2 a, D2 b) { return mul(madd(rl, a, mul(rr, b)), ir); };
      const D2 ul = r.E(1, k), ur = r.E(1, k + S);
      D2 tl{}, tr{};
      un = mean(ul, ur);
      if constexpr (T::M == 4) {
        tl = r.E(3, k);
        tr = r.E(3, k + S);
        ut = mean(tl, tr);
      }
      using C = LineChar<D2, T::M, 0>;
      const D2 q = sub(mean(C::kinetic(ul, tl), C::kinetic(ur, tr)), C::kinetic(un, ut));
      H = madd(gm1(), q, mean(r.E(2, k), r.E(2, k + S)));
      return;
    }
    const D2 is = div(D2{1.f, 0.f}, add(sl, sr));
    auto roe = [&](int e) { return mul(madd(sl, r.E(e, k), mul(sr, r.E(e, k + S))), is); };
    un = roe(1);
    H = roe(2);
    if constexpr (T::M == 4) ut = roe(3);
  }
};
template <class T, bool ROWS>
struct LineData<double, T, ROWS> {
  const T& r;
  int S;
  double alpha, dx;
  const SchemeParams& sp;
  __device__ __forceinline__ LineData(const T& r_, int S_, double al, double d,
                                      const SchemeParams& sp_)
      : r(r_), S(S_), alpha(al), dx(d), sp(sp_) {}
  __device__ __forceinline__ double H(int sd, int c, int k) const {
    if constexpr (ROWS) return r.pd(sd * T::M + c, k);
    return mul(0.5 * dx, madd(alpha, r.N(c, k), sd ? -r.h(c, k) : r.h(c, k)));
  }
  __device__ __forceinline__ double X(int sd, int c, int k) const {
    if constexpr (ROWS) return r.pd((2 + sd) * T::M + c, k);
    const double dF = sub(r.F(c, k + S), r.F(c, k));
    return mul(0.5, madd(alpha, dU(c, k), sd ? -dF : dF));
  }
  __device__ __forceinline__ double dU(int c, int k) const {
    return sub(r.U(c, k + S), r.U(c, k));
  }
  __device__ __forceinline__ double Nx(int c, int k) const { return mul(dx, r.N(c, k)); }
  __device__ __forceinline__ double gm1() const { return sp.wd[9] - 1.0; }
  __device__ __forceinline__ void prim(const double* u, double& un, double& ut, double& H) const {
    constexpr int M = T::M, kn = T::kn, kt = 3 - T::kn;
    const double ir = recip_fp64(u[0]);
    un = mul(u[kn], ir);
    double ke = mul(u[kn], un);
    if constexpr (M == 4) {
      ut = mul(u[kt], ir);
      ke = madd(u[kt], ut, ke);
    }
    H = mul(madd(gm1(), madd(-0.5, ke, u[M - 1]), u[M - 1]), ir);
  }
  // the rows of the eigen-system's inputs (LineTile::E)
  static constexpr int kE = (T::SLIM ? 4 : 6) * T::M;
  // point k's velocities and enthalpy
  __device__ __forceinline__ void prim_at(int k, double& un, double& ut, double& H) const {
    if constexpr (ROWS) {
      un = r.pd(kE + 1, k);
      H = r.pd(kE + 2, k);
      if constexpr (T::M == 4) ut = r.pd(kE + 3, k);
      return;
    }
    double a[T::M];
#pragma unroll
    for (int c = 0; c < T::M; ++c) a[c] = r.U(c, k);
    prim(a, un, ut, H);
  }
  // sqrt(rho)
  __device__ __forceinline__ double root(int k) const {
    if constexpr (ROWS) return r.pd(kE, k);
    return mul(r.U(0, k), rsqrt_fp64(r.U(0, k)));
  }
  __device__ __forceinline__ void state(int k, bool edge, double& un, double& ut, double& H) const {
    if (!edge) {
      prim_at(k, un, ut, H);
    } else if (sp.eig_avg == 0) {  // Roe average
      double uL, tL = 0.0, HL, uR, tR = 0.0, HR;
      prim_at(k, uL, tL, HL);
      prim_at(k + S, uR, tR, HR);
      const double sl = root(k), sr = root(k + S), is = recip_fp64(add(sl, sr));
      auto roe = [&](double x, double y) { return mul(add(mul(sl, x), mul(sr, y)), is); };
      un = roe(uL, uR);
      ut = roe(tL, tR);
      H = roe(HL, HR);
    } else {  // arithmetic mean state
      double a[T::M];
#pragma unroll
      for (int c = 0; c < T::M; ++c) a[c] = mul(0.5, add(r.U(c, k), r.U(c, k + S)));
      prim(a, un, ut, H);
    }
  }
};

// Makes of the pair rows doubles of the same quantities, bit for bit what
// LineData<double, T> forms on the fly: once per point and edge instead of by
// every item that reads them (Euler: about 160 of 1050 FP64 instructions per
// point where all items are listed; rhs of such a batch of 614 k points 1296 ->
// 1122 us). For tiles with many listed items, when the
// pairs are no longer needed; followed by a barrier.
template <class T>
__device__ __forceinline__ void double_rows(const T& r, int S, double alpha, double dx,
                                            const SchemeParams& sp) {
  constexpr int M = T::M;
  const LineData<double, T> in(r, S, alpha, dx, sp);
  for (int k = threadIdx.x; k < r.L; k += blockDim.x) {
#pragma unroll
    for (int c = 0; c < M; ++c) {
      r.pd(c, k) = in.H(0, c, k);
      r.pd(M + c, k) = in.H(1, c, k);
    }
    if constexpr (T::EUL) {
      double un, ut = 0.0, H;
      in.prim_at(k, un, ut, H);
      r.pd(in.kE, k) = in.root(k);
      r.pd(in.kE + 1, k) = un;
      r.pd(in.kE + 2, k) = H;
      if constexpr (M == 4) r.pd(in.kE + 3, k) = ut;
    }
    if (k + S < r.L) {
#pragma unroll
      for (int c = 0; c < M; ++c) {
        r.pd(2 * M + c, k) = in.X(0, c, k);
        r.pd(3 * M + c, k) = in.X(1, c, k);
      }
    }
  }
}

// c ? a + y : a
template <class X>
__device__ __forceinline__ X add_if(bool c, X a, X y) {
  return add(a, pick2(c, y, X{}));
}

// The stencil differences of side sd of the interface between k and k + S,
// component c (the arguments of side_correction): the "+" side is about point
// k, the "-" side about k + S. The latter reverses the stencil and negates H;
// with -H^- and -M for H^+ and P (M the difference of f^- along an edge) its
// expressions are those of the "+" side.
template <class X, class T, bool R>
__device__ __forceinline__ void side_differences(const LineData<X, T, R>& in, int sd, int c, int k,
                                                 int S, X* x) {
  using P2 = typename Num<X>::Scale;
  const int k0 = sd ? k + S : k, km = sd ? k0 + S : k0 - S, kp = sd ? k : k0 + S;
  // the edges (k - S, k), (k, k + S) or (k + S, k + 2 S), (k, k + S)
  const X Hm = in.H(sd, c, km), H0 = in.H(sd, c, k0), Hp = in.H(sd, c, kp);
  x[0] = sub(H0, in.X(sd, c, sd ? k0 : km));
  x[1] = sub(H0, in.X(sd, c, k));
  x[2] = scale_add(H0, P2(-2), add(Hm, Hp));
  x[3] = sub(Hm, Hp);
  x[4] = H0;
}
// Both sides packed.
template <class T>
__device__ __forceinline__ void sides_differences(const LineData<D2, T>& in, int c, int k, int S,
                                                  Q2* x) {
  auto at = [&](int a, int b) { return both(in.H(0, c, a), in.H(1, c, b)); };
  const Q2 Hm = at(k - S, k + 2 * S), H0 = at(k, k + S), Hp = at(k + S, k);
  x[0] = sub(H0, both(in.X(0, c, k - S), in.X(1, c, k + S)));
  x[1] = sub(H0, both(in.X(0, c, k), in.X(1, c, k)));
  x[2] = scale_add(H0, -2.f, add(Hm, Hp));
  x[3] = sub(Hm, Hp);
  x[4] = H0;
}

template <class T, class X, int DIR>
using CharOf = LineChar<X, T::M == 1 ? 3 : T::M, T::M == 1 ? 0 : DIR>;

// The characteristic system of the interface between k and k + S (`edge`) or
// of point k.
template <int DIR, class X, class T, bool R>
__device__ __forceinline__ CharOf<T, X, DIR> char_system(const LineData<X, T, R>& in, int k,
                                                         bool edge) {
  CharOf<T, X, DIR> ch;
  if constexpr (T::EUL) {
    X un, ut{}, H;
    in.state(k, edge, un, ut, H);
    const X q = ch.kinetic(un, ut);
    ch.init(un, ut, H, q, mul(in.gm1(), sub(H, q)), in.gm1());
  }
  return ch;
}

// Adds side sd of the interface between k and k + S to the characteristic
// fields f (pairs: 12 times the corrections; FP64: the side's values) and, in
// pairs, to 60 times the linear parts; returns, in pairs, 12 times the sum of
// the fields' bounds of side_correction in units of the density. ONE: field
// q0 alone, to f[0].
template <int DIR, bool ONE = false, class X, class T, bool R>
__device__ __forceinline__ float interface_side(const LineData<X, T, R>& in,
                                                const CharOf<T, X, DIR>& ch,
                                                const LineWeights<X>& w, int sd, int k, int S,
                                                X* f, X* lin, int q0 = 0) {
  constexpr int M = T::M;
  constexpr bool FP64 = std::is_same<X, double>::value;
  float sum = 0.f;
  auto side = [&](int q, X y1, X y2, X s, X d, X H0) {
    if constexpr (FP64) {
      return side_value(y1, y2, s, d, H0, w);
    } else {
      float e = 0.f;
      const D2 v = side_correction(y1, y2, s, d, H0, w, e);
      sum += T::EUL ? ch.density_units(q, e) : e;
      return v;
    }
  };
  X x[M][5];
#pragma unroll
  for (int c = 0; c < M; ++c) {
    side_differences(in, sd, c, k, S, x[c]);
    if constexpr (!FP64) lin[c] = add(lin[c], linear_part(x[c][0], x[c][1], x[c][3]));
  }
  if constexpr (T::EUL) {
    typename CharOf<T, X, DIR>::Factors a[5];
#pragma unroll
    for (int v = 0; v < 5; ++v) {
      X y[M];
#pragma unroll
      for (int c = 0; c < M; ++c) y[c] = x[c][v];
      a[v] = ch.factors(y);
    }
    if constexpr (ONE) {
      f[0] = side(q0, a[0].field(q0), a[1].field(q0), a[2].field(q0), a[3].field(q0),
                  a[4].field(q0));
      return sum;
    }
#pragma unroll 1
    for (int q = 0; q < M; ++q) {
      const X y = side(q, a[0].field(q), a[1].field(q), a[2].field(q), a[3].field(q),
                       a[4].field(q));
#pragma unroll
      for (int c = 0; c < M; ++c) f[c] = add_if(q == c, f[c], y);
    }
  } else {
    f[0] = add(f[0], side(0, x[0][0], x[0][1], x[0][2], x[0][3], x[0][4]));
  }
  return sum;
}

// Whether the interface between k and k + S, of whose bounds `e` is the sum
// over both sides, may be taken in pairs: e = 0, or small against alpha times
// the smaller of the two densities (scalar equations: values).
template <class T>
__device__ __forceinline__ bool interface_weak(const T& r, int k, int S, float e, double alpha,
                                               const SchemeParams& sp) {
  float level;
  if constexpr (T::EUL) {
    const float s = fminf(r.E(0, k).h, r.E(0, k + S).h);
    level = s * s;
  } else {
    level = fminf(fabsf(to_float(r.U(0, k))), fabsf(to_float(r.U(0, k + S))));
  }
  // (false for a NaN: of e, or of a level or alpha outside the pairs' range)
  return e <= 12.f * (T::EUL ? kWeakLevel : kWeakScalar) * scale_pair(alpha).h * level;
}

// Leading words: the largest of component c at the edges and points that the
// interface between k and k + S takes its differences from.
template <class T>
__device__ __forceinline__ float difference_top(const LineData<D2, T>& in, int c, int k, int S) {
  auto top = [](D2 a, D2 b) { return fmaxf(fabsf(a.h), fabsf(b.h)); };
  return fmaxf(top(in.H(0, c, k), in.H(1, c, k + S)),
               fmaxf(top(in.X(0, c, k), in.X(1, c, k)), top(in.X(0, c, k - S), in.X(1, c, k + S))));
}
// The largest of a vector's components in units of the density: momenta over
// sqrt(H), the energy over H (an enthalpy near the point).
template <class T>
__device__ __forceinline__ float in_density(const float* x, float H) {
  float m = fabsf(x[T::kn]);
  if constexpr (T::M == 4) m = fmaxf(m, fabsf(x[3 - T::kn]));
  return fmaxf(fabsf(x[0]), fmaxf(m * rsqrtf(H), fabsf(x[T::M - 1]) * fast_rcp(H)));
}

// How the interface between k and k + S is evaluated, decided before any of the
// work. `pairs`: tried in pairs; `linear`: with the linear part in pairs, which
// has an error of 2^-48 of the differences it is made of (in FP64: one of F's
// rounding). Euler tries only interfaces whose differences are at most kFine
// of alpha U, where the linear part's and the derivative flux's errors stay
// below the FP64 form's (1/16: up to 1.08 of it, 1/32: 0.6). Scalar equations
// take the linear part in FP64 where a difference exceeds 2^-3 of F (coarse
// grids, sonic points; error of L^1 over the FP64 form's: wave of 15 points
// 4.2 -> 0.4). All their interfaces are tried: a test for those that would be
// listed afterwards cost the Buckley-Leverett batch 6% and took 1% off a flow
// of noise. None is tried where alpha or the density leaves the pairs' range.
struct Route {
  bool pairs, linear;
};
constexpr float kFine = 1.f / 20.f;
template <class T>
__device__ __forceinline__ Route interface_route(const LineData<D2, T>& in, int k, int S,
                                                 double alpha) {
  const float al = scale_pair(alpha).h;
  if constexpr (T::EUL) {
    const float s = fminf(in.r.E(0, k).h, in.r.E(0, k + S).h);
    float x[T::M];
#pragma unroll
    for (int c = 0; c < T::M; ++c) x[c] = difference_top(in, c, k, S);
    const float H = fminf(in.r.E(2, k).h, in.r.E(2, k + S).h);
    // (x[0] by itself: fmaxf would drop a NaN)
    return Route{x[0] <= kFine * al * s * s && in_density<T>(x, H) <= kFine * al * s * s, true};
  } else {
    auto larger = [&](double a, double b) { return fmaxf(fabsf(to_float(a)), fabsf(to_float(b))); };
    const float top = fmaxf(fmaxf(fabsf(in.H(0, 0, k).h), fabsf(in.H(1, 0, k + S).h)),
                            fmaxf(fabsf(in.X(0, 0, k).h), fabsf(in.X(1, 0, k).h)));
    return Route{al > 0.f, top <= 0x1p-3f * larger(in.r.F(0, k), in.r.F(0, k + S))};
  }
}
// Whether the limiter's point k is tried in pairs, from the second differences (in units of
// the density, the component's own): not where they exceed 1/16 of the density,
// or a quarter of the first differences, and tau's unit.
template <class T>
__device__ __forceinline__ bool limiter_fine(const LineData<D2, T>& in, int k, int S) {
  const T& r = in.r;
  const float g = fmaxf(in.sp.wp[4].h, in.sp.wp[5].h);
  float lap[T::M];
  bool fine = true;
#pragma unroll
  for (int c = 0; c < T::M; ++c) {
    const float q1 = r.dU_lead(c, k - S), q2 = r.dU_lead(c, k);
    lap[c] = q2 - q1;
    fine &= fabsf(lap[c]) <= 0.25f * (fabsf(q1) + fabsf(q2)) || g * lap[c] * lap[c] < 0x1p-14f;
  }
  if constexpr (T::EUL) {
    if (in.sp.limiter != 2) {
      const float s = r.E(0, k).h, x = in_density<T>(lap, r.E(2, k).h);
      fine = x <= 0.0625f * s * s || g * x * x < 0x1p-14f;
    }
  }
  return fine;
}

// The linear part of the scalar c in FP64.
template <class T>
__device__ __forceinline__ double linear_part_fp64(const T& r, int k, int S, double alpha,
                                                   double dx) {
  const int m = k - S, p = k + S, q = k + 2 * S;
  const double h = madd(33.0, sub(r.h(0, k), r.h(0, p)), mul(3.0, sub(r.h(0, m), r.h(0, q))));
  const double N = madd(27.0, add(r.N(0, k), r.N(0, p)), mul(3.0, add(r.N(0, m), r.N(0, q))));
  const double F = sub(sub(r.F(0, q), r.F(0, p)), sub(r.F(0, k), r.F(0, m)));
  const double U = madd(27.0, sub(r.U(0, p), r.U(0, k)), mul(11.0, sub(r.U(0, q), r.U(0, m))));
  const double x = madd(11.0, F, mul(alpha, madd(dx, N, -U)));
  return mul(1.0 / 120.0, madd(dx, h, x));
}

// c from the sums over both sides (lin64: the scalar linear part, where
// `linear` is false).
template <int DIR, class X, class T, bool R>
__device__ __forceinline__ void interface_value(const LineData<X, T, R>& in,
                                                const CharOf<T, X, DIR>& ch, int k, int S,
                                                double alpha, X* f, const X* lin, bool linear,
                                                double lin64, double* cc) {
  constexpr int M = T::M;
  if constexpr (T::EUL) {
    X out[M];
    ch.right(f, out);
#pragma unroll
    for (int c = 0; c < M; ++c) f[c] = out[c];
  }
#pragma unroll
  for (int c = 0; c < M; ++c) {
    // f^+_i + f^-_{i+1} = (F_i + F_{i+1}) / 2 - alpha (U_{i+1} - U_i) / 2
    if constexpr (std::is_same<X, double>::value)
      cc[c] = madd(-0.5 * alpha, in.dU(c, k), f[c]);
    else
      cc[c] = to_double(madd(dconst(1.0 / 60.0), lin[c], mul(f[c], dconst(1.0 / 12.0))));
  }
  if constexpr (!T::EUL && std::is_same<X, D2>::value)
    if (!linear) cc[0] = add(lin64, to_double(mul(f[0], dconst(1.0 / 12.0))));
}

// The derivative flux dx (h-hat^+ + h-hat^-) of component c at the interface
// between k and k + S: both sides' p_0' of Sec. 2.1 in terms of F, U, h, N.
template <class T>
__device__ __forceinline__ double derivative_flux_fp64(const T& r, int c, int k, int S,
                                                       double alpha, double dx) {
  const double kU = mul(0.125, alpha), kh = mul(dx, 1.0 / 24.0), kv = mul(alpha, kh);
  const int m = k - S, p = k + S, q = k + 2 * S;
  const double t0 = sub(r.F(c, p), r.F(c, k)), t1 = sub(r.F(c, q), r.F(c, m));
  const double su = sub(sub(r.U(c, q), r.U(c, p)), sub(r.U(c, k), r.U(c, m)));
  const double sh = madd(-7.0, add(r.h(c, k), r.h(c, p)), add(r.h(c, m), r.h(c, q)));
  const double sv = madd(3.0, sub(r.N(c, k), r.N(c, p)), sub(r.N(c, m), r.N(c, q)));
  return madd(1.875, t0, madd(-0.125, t1, madd(kU, su, madd(kh, sh, mul(kv, sv)))));
}

// The same from both sides' differences: Euler in pairs (45 fewer FP64
// instructions per point and stage of 1D: batch of Riemann problems 7.52 ->
// 6.74 ms); scalar equations in FP64, where the pairs' error was up to twice
// that on grids of less than 100 points.
template <class T>
__device__ __forceinline__ double derivative_flux(const LineData<D2, T>& in, const Q2* x, int c,
                                                  int k, int S, double alpha, double dx) {
  if constexpr (!T::EUL) return derivative_flux_fp64(in.r, c, k, S, alpha, dx);
  const Q2 d = derivative_part(x[0], x[1], x[2], x[3], x[4]);
  return to_double(scale(sub(first(d), second(d)), 0.25f));
}

// Both sides as interface_side, packed: the same operations on the two lanes.
template <int DIR, class T>
__device__ __forceinline__ float interface_sides(const LineData<D2, T>& in,
                                                 const CharOf<T, D2, DIR>& ch,
                                                 const LineWeights<D2>& w_, int k, int S, D2* f,
                                                 D2* lin, double alpha, double dx, double* dd) {
  constexpr int M = T::M;
  const LineWeights<Q2> w{both(w_.g0), both(w_.g1), both(w_.g2), both(w_.eps), w_.bmax};
  float2 sum = make_float2(0.f, 0.f);
  auto sides = [&](int q, Q2 y1, Q2 y2, Q2 s, Q2 d, Q2 H0) {
    float2 e = make_float2(0.f, 0.f);
    const Q2 v = side_correction(y1, y2, s, d, H0, w, e);
    sum.x += T::EUL ? ch.density_units(q, e.x) : e.x;
    sum.y += T::EUL ? ch.density_units(q, e.y) : e.y;
    return add(first(v), second(v));
  };
  Q2 x[M][5];
#pragma unroll
  for (int c = 0; c < M; ++c) {
    sides_differences(in, c, k, S, x[c]);
    const Q2 l = linear_part(x[c][0], x[c][1], x[c][3]);
    lin[c] = add(first(l), second(l));
    dd[c] = derivative_flux(in, x[c], c, k, S, alpha, dx);
  }
  if constexpr (T::EUL) {
    const auto chq = ch.packed();
    typename LineChar<Q2, M, DIR>::Factors a[5];
#pragma unroll
    for (int v = 0; v < 5; ++v) {
      Q2 y[M];
#pragma unroll
      for (int c = 0; c < M; ++c) y[c] = x[c][v];
      a[v] = chq.factors(y);
    }
#pragma unroll
    for (int c = 0; c < M; ++c) f[c] = D2{0.f, 0.f};
#pragma unroll kUnrollFields
    for (int q = 0; q < M; ++q) {
      const D2 y = sides(q, a[0].field(q), a[1].field(q), a[2].field(q), a[3].field(q),
                         a[4].field(q));
#pragma unroll
      for (int c = 0; c < M; ++c) f[c] = pick2(q == c, y, f[c]);
    }
  } else {
    f[0] = sides(0, x[0][0], x[0][1], x[0][2], x[0][3], x[0][4]);
  }
  return sum.x + sum.y;
}

// c (to cc) and, in pairs, the derivative flux (to dd) of the interface between
// points k and k + S; in pairs, false when the correction is not small (the
// values are then not to be used).
template <class X, int DIR, bool ROWS = false, class T>
__device__ __forceinline__ bool interface_line(const T& r, int k, int S, double alpha, double dx,
                                               const SchemeParams& sp, double* cc,
                                               double* dd = nullptr) {
  const LineData<X, T, ROWS> in(r, S, alpha, dx, sp);
  Route route{true, true};
  if constexpr (!std::is_same<X, double>::value) {
    route = interface_route(in, k, S, alpha);
    if (!route.pairs) {
#pragma unroll
      for (int c = 0; c < T::M; ++c) cc[c] = dd[c] = 0.0;
      return false;
    }
  }
  const LineWeights<X> w = line_weights<X>(sp, false);
  const auto ch = char_system<DIR>(in, k, true);
  X f[T::M], lin[T::M];
  if constexpr (std::is_same<X, double>::value) {
#pragma unroll
    for (int c = 0; c < T::M; ++c) f[c] = lin[c] = X{};
#pragma unroll 1
    for (int sd = 0; sd < 2; ++sd) interface_side<DIR>(in, ch, w, sd, k, S, f, lin);
    interface_value<DIR>(in, ch, k, S, alpha, f, lin, true, 0.0, cc);
    return true;
  } else {
    const float e = interface_sides<DIR>(in, ch, w, k, S, f, lin, alpha, dx, dd);
    const bool weak = interface_weak(r, k, S, e, alpha, sp);
    double lin64 = 0.0;
    if (weak && !route.linear) lin64 = linear_part_fp64(r, k, S, alpha, dx);
    interface_value<DIR>(in, ch, k, S, alpha, f, lin, route.linear, lin64, cc);
    return weak;
  }
}

// The limiter's four differences at point k, component c.
template <class X, class T, bool R>
__device__ __forceinline__ void limiter_differences(const LineData<X, T, R>& in, int c, int k, int S,
                                                    X* x) {
  x[0] = in.dU(c, k - S);
  x[1] = in.dU(c, k);
  x[2] = in.Nx(c, k - S);
  x[3] = in.Nx(c, k + S);
}

// The limited derivative from its characteristic fields (chars) or
// components z: pairs, 4 times the corrections to the linear
// dx q_0' = 3/4 (u_{i+1} - u_{i-1}) - dx (v_{i-1} + v_{i+1}) / 4; FP64, dx v~.
template <int DIR, class X, class T, bool R>
__device__ __forceinline__ void limiter_sum(const LineData<X, T, R>& in, const CharOf<T, X, DIR>& ch,
                                            int k, int S, double idx, bool chars, X* z,
                                            double* vt) {
  constexpr int M = T::M;
  const T& r = in.r;
  if constexpr (T::EUL) {
    if (chars) {
      X out[M];
      ch.right(z, out);
#pragma unroll
      for (int c = 0; c < M; ++c) z[c] = out[c];
    }
  }
  const double k3 = mul(0.75, idx), k1 = mul(0.25, idx);
#pragma unroll
  for (int c = 0; c < M; ++c) {
    if constexpr (std::is_same<X, double>::value) {
      vt[c] = mul(idx, z[c]);
    } else {
      const double q0 = madd(k3, sub(r.U(c, k + S), r.U(c, k - S)),
                             mul(-0.25, add(r.N(c, k - S), r.N(c, k + S))));
      vt[c] = madd(k1, to_double(z[c].l), madd(k1, to_double(z[c].h), q0));
    }
  }
}

// Characteristic field (or component) q of the limiter at point k in pairs,
// with the characteristic system it makes for limiter_sum.
template <int DIR, class T>
__device__ __forceinline__ D2 limiter_field(const LineData<D2, T>& in, CharOf<T, D2, DIR>& ch,
                                            int k, int S, const SchemeParams& sp, int q,
                                            float& e) {
  constexpr int M = T::M;
  D2 y[4];
  if (T::EUL && sp.limiter != 2) {  // uniform
    if constexpr (T::EUL) {
      D2 x[M][4];
#pragma unroll
      for (int c = 0; c < M; ++c) limiter_differences(in, c, k, S, x[c]);
      ch = char_system<DIR>(in, k, false);
#pragma unroll
      for (int v = 0; v < 4; ++v) {
        D2 u[M];
#pragma unroll
        for (int c = 0; c < M; ++c) u[c] = x[c][v];
        y[v] = ch.factors(u).field(q);
      }
    }
  } else {
    limiter_differences(in, q, k, S, y);
  }
  const D2 z = limiter_correction(y[0], y[1], y[2], y[3], line_weights<D2>(sp, true), e);
  if (T::EUL && sp.limiter != 2) e = ch.density_units(q, e);
  return z;
}

// Whether point k's limited derivative, of whose bounds `e` is the sum, may be
// taken in pairs: e = 0, or (characteristic fields, whose FP64 form starts
// from projected values) small against the density.
template <class T>
__device__ __forceinline__ bool limiter_weak(const T& r, int k, float e, const SchemeParams& sp) {
  if constexpr (T::EUL) {
    if (sp.limiter != 2) {
      const float s = r.E(0, k).h;
      return e <= 4.f * kWeakLimiter * s * s;
    }
  }
  return e <= 0.f;
}

// The limited derivative at point k; in pairs, false as interface_line.
template <class X, int DIR, bool ROWS = false, class T>
__device__ __forceinline__ bool limiter_line(const T& r, int k, int S, double dx, double idx,
                                             const SchemeParams& sp, double* vt) {
  constexpr int M = T::M;
  const LineData<X, T, ROWS> in(r, S, 0.0, dx, sp);
  if constexpr (!std::is_same<X, double>::value) {
    if (!limiter_fine(in, k, S)) {
#pragma unroll
      for (int c = 0; c < M; ++c) vt[c] = 0.0;
      return false;
    }
  }
  float sum = 0.f;
  X x[M][4], z[M];
#pragma unroll
  for (int c = 0; c < M; ++c) limiter_differences(in, c, k, S, x[c]);
  const LineWeights<X> w = line_weights<X>(sp, true);
  const bool chars = T::EUL && sp.limiter != 2;  // uniform
  CharOf<T, X, DIR> ch;
  auto limit = [&](int q, X q1, X q2, X Vm, X Vp) {
    if constexpr (std::is_same<X, double>::value) {
      return limiter_value(q1, q2, Vm, Vp, w);
    } else {
      float e = 0.f;
      const D2 v = limiter_correction(q1, q2, Vm, Vp, w, e);
      sum += chars ? ch.density_units(q, e) : e;
      return v;
    }
  };
  if (chars) {
    if constexpr (T::EUL) {
      ch = char_system<DIR>(in, k, false);
      typename CharOf<T, X, DIR>::Factors a[4];
#pragma unroll
      for (int v = 0; v < 4; ++v) {
        X y[M];
#pragma unroll
        for (int c = 0; c < M; ++c) y[c] = x[c][v];
        a[v] = ch.factors(y);
      }
#pragma unroll
      for (int c = 0; c < M; ++c) z[c] = X{};
      if constexpr (std::is_same<X, double>::value) {
#pragma unroll 1
        for (int q = 0; q < M; ++q) {
          const X y = limit(q, a[0].field(q), a[1].field(q), a[2].field(q), a[3].field(q));
#pragma unroll
          for (int c = 0; c < M; ++c) z[c] = pick2(q == c, y, z[c]);
        }
      } else {  // two fields packed (three fields: the last one twice)
        const LineWeights<Q2> wq{both(w.g0), both(w.g1), both(w.g2), both(w.eps), w.bmax};
#pragma unroll kUnrollFields
        for (int h = 0; h < 2; ++h) {
          const int qa = 2 * h, qb = M == 3 && h == 1 ? 2 : qa + 1;
          auto two = [&](int v) { return both(a[v].field(qa), a[v].field(qb)); };
          float2 e = make_float2(0.f, 0.f);
          const Q2 y = limiter_correction(two(0), two(1), two(2), two(3), wq, e);
          sum += ch.density_units(qa, e.x);
          if (qb != qa) sum += ch.density_units(qb, e.y);
#pragma unroll
          for (int c = 0; c < M; ++c)
            z[c] = pick2(c == qa, first(y), pick2(c == qb, second(y), z[c]));
        }
      }
    }
  } else {
#pragma unroll
    for (int c = 0; c < M; ++c) z[c] = limit(c, x[c][0], x[c][1], x[c][2], x[c][3]);
  }
  limiter_sum<DIR>(in, ch, k, S, idx, chars, z, vt);
  if constexpr (std::is_same<X, double>::value) return true;
  else return limiter_weak(r, k, sum, sp);
}

// ---------------------------------------------------------------------------
// The same items in FP64 with the work of one item divided over a group of
// lanes (an FP64 warp instruction costs the same however many lanes are
// active, so a few items are done sooner the fewer instructions each lane
// has): lane (sd, c) of an interface's group forms the stencil differences of
// side sd for component c and, after an exchange, evaluates field c of that
// side. About 150 FP64 instructions per warp of four interfaces (Euler),
// against 450 per warp of up to 32 in interface_line.
// ---------------------------------------------------------------------------
template <class T>
struct Group {
  static constexpr int NC = T::M == 1 ? 1 : 4;  // lanes per side
  static constexpr int kInterface = 2 * NC, kPoint = NC;  // lanes per item
  // FP64 instructions of a warp of items: in groups, and one item per thread
  static constexpr int group_f = T::M == 1 ? 75 : 150, whole_f = T::M == 1 ? 130 : 450;
  static constexpr int group_l = T::M == 1 ? 60 : 115, whole_l = T::M == 1 ? 60 : 300;
  // Whether n items are sooner done in groups: the FP64 pipes of an SM's four
  // sub-partitions set the time, however many warps share them. (With the
  // warps of the CTA for the four, the wide form's 16 took a whole tile of
  // listed items in groups: rhs of an Euler instance of 200 points, all items
  // listed, 92 us; with this rule and double_rows 53.)
  __host__ __device__ static constexpr bool few(int n, int lanes, int group, int whole) {
    const int per = 32 / lanes;
    return ((n + per - 1) / per + 3) / 4 * group <= ((n + 31) / 32 + 3) / 4 * whole;
  }
};

// c of the interface (k, k + S), output index j, by the lanes of a group;
// `live` false: the lanes take part without an item (k any valid index).
template <int DIR, class T>
__device__ __forceinline__ void interface_group(const T& r, int k, int S, int j, bool live,
                                                double alpha, double dx, const SchemeParams& sp) {
  constexpr int M = T::M, NC = Group<T>::NC;
  constexpr unsigned all = 0xffffffffu;
  const int lane = threadIdx.x & 31, sd = lane / NC & 1, q = lane & (NC - 1);
  const int c = q < M ? q : 0, first = lane - q;  // this side's lanes
  const LineData<double, T> in(r, S, alpha, dx, sp);
  const LineWeights<double> w = line_weights<double>(sp, false);
  LineChar<double, M == 1 ? 3 : M, M == 1 ? 0 : DIR> ch;
  if constexpr (T::EUL) {
    double un, ut = 0.0, H;
    if (sp.eig_avg == 0) {  // Roe average; each side's lanes take one state
      const int ks = sd ? k + S : k;
      in.prim_at(ks, un, ut, H);
      const double s = mul(r.U(0, ks), rsqrt_fp64(r.U(0, ks)));
      const double so = __shfl_xor_sync(all, s, NC), is = recip_fp64(add(s, so));
      auto roe = [&](double x) {
        const double m = mul(s, x), o = __shfl_xor_sync(all, m, NC);
        return mul(add(m, o), is);
      };
      un = roe(un);
      H = roe(H);
      if constexpr (M == 4) ut = roe(ut);
    } else {
      in.state(k, true, un, ut, H);
    }
    const double kin = ch.kinetic(un, ut);
    ch.init(un, ut, H, kin, mul(in.gm1(), sub(H, kin)), in.gm1());
  }
  double x[5];
  side_differences(in, sd, c, k, S, x);
  if constexpr (T::EUL) {
    typename decltype(ch)::Factors a[5];
#pragma unroll
    for (int v = 0; v < 5; ++v) {
      double y[M];
#pragma unroll
      for (int i = 0; i < M; ++i) y[i] = __shfl_sync(all, x[v], first + i);
      a[v] = ch.factors(y);
    }
#pragma unroll
    for (int v = 0; v < 5; ++v) x[v] = a[v].field(c);
  }
  double f = side_value(x[0], x[1], x[2], x[3], x[4], w);
  f = add(f, __shfl_xor_sync(all, f, NC));
  if constexpr (T::EUL) {
    double g[M], out[M];
#pragma unroll
    for (int i = 0; i < M; ++i) g[i] = __shfl_sync(all, f, first + i);
    ch.right(g, out);
    f = out[0];
#pragma unroll
    for (int i = 1; i < M; ++i) f = c == i ? out[i] : f;
  }
  if (live && sd == 0 && q < M) r.C(c, j) = madd(-0.5 * alpha, in.dU(c, k), f);
}

// The limited derivative at point k, output index j, lane c of a group for
// component and field c.
template <int DIR, class T>
__device__ __forceinline__ void limiter_group(const T& r, int k, int S, int j, bool live,
                                              double dx, double idx, const SchemeParams& sp) {
  constexpr int M = T::M, NC = Group<T>::NC;
  constexpr unsigned all = 0xffffffffu;
  const int lane = threadIdx.x & 31, q = lane & (NC - 1);
  const int c = q < M ? q : 0, first = lane - q;
  const LineData<double, T> in(r, S, 0.0, dx, sp);
  const LineWeights<double> w = line_weights<double>(sp, true);
  double x[4] = {in.dU(c, k - S), in.dU(c, k), in.Nx(c, k - S), in.Nx(c, k + S)};
  double z;
  if (T::EUL && sp.limiter != 2) {  // uniform
    if constexpr (T::EUL) {
      const auto ch = char_system<DIR>(in, k, false);
#pragma unroll
      for (int v = 0; v < 4; ++v) {
        double y[M];
#pragma unroll
        for (int i = 0; i < M; ++i) y[i] = __shfl_sync(all, x[v], first + i);
        x[v] = ch.factors(y).field(c);
      }
      z = limiter_value(x[0], x[1], x[2], x[3], w);
      double g[M], out[M];
#pragma unroll
      for (int i = 0; i < M; ++i) g[i] = __shfl_sync(all, z, first + i);
      ch.right(g, out);
      z = out[0];
#pragma unroll
      for (int i = 1; i < M; ++i) z = c == i ? out[i] : z;
    }
  } else {
    z = limiter_value(x[0], x[1], x[2], x[3], w);
  }
  if (live && q < M) r.lim(c, j) = mul(idx, z);
}

// Evaluates a tile's listed interfaces and points in FP64: few by groups of
// lanes, their groups dealt to the CTA's warps (the first one differing from
// tile to tile), many by one thread each. at(j, lim) gives the flat index of
// interface or point j. Both ways give the same bits (the arithmetic is the
// same, without contraction), so that a point's result does not depend on its
// tile. Every thread of the CTA calls it; the results are visible after the
// next barrier.
template <int DIR, class T, class At>
__device__ __forceinline__ void listed_items(const T& r, const unsigned short* list_f, int nf,
                                             const unsigned short* list_l, int nl, At at, int S,
                                             int rot, double alpha, double dx, double idx,
                                             const SchemeParams& sp) {
  constexpr int M = T::M;
  using G = Group<T>;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  constexpr int gf = 32 / G::kInterface, gl = 32 / G::kPoint;
  const bool few_f = G::few(nf, G::kInterface, G::group_f, G::whole_f);
  const bool few_l = G::few(nl, G::kPoint, G::group_l, G::whole_l);
  if (!few_f || !few_l) {  // uniform
    double_rows(r, S, alpha, dx, sp);
    __syncthreads();
  }
  const int uf = few_f ? (nf + gf - 1) / gf : (nf + 31) / 32;
  const int ul = few_l ? (nl + gl - 1) / gl : (nl + 31) / 32;
  // Euler: the listed interfaces' derivative fluxes, a component per lane
  const int ud = T::EUL ? (nf * M + 31) / 32 : 0;
  for (int u = (warp + rot) % nw; u < uf + ul + ud; u += nw) {
    if (u >= uf + ul) {
      const int i = (u - uf - ul) * 32 + lane;
      if (i < nf * M) {
        const int j = list_f[i / M];
        r.D(i % M, j) = derivative_flux_fp64(r, i % M, at(j, false), S, alpha, dx);
      }
    } else if (u < uf) {
      if (few_f) {
        const int i = u * gf + lane / G::kInterface;
        const bool live = i < nf;
        const int j = list_f[live ? i : 0];
        interface_group<DIR>(r, at(j, false), S, j, live, alpha, dx, sp);
      } else if (u * 32 + lane < nf) {
        const int j = list_f[u * 32 + lane];
        double x[M];
        interface_line<double, DIR, true>(r, at(j, false), S, alpha, dx, sp, x);
#pragma unroll
        for (int c = 0; c < M; ++c) r.C(c, j) = x[c];
      }
    } else {
      const int v = u - uf;
      if (few_l) {
        const int i = v * gl + lane / G::kPoint;
        const bool live = i < nl;
        const int j = list_l[live ? i : 0];
        limiter_group<DIR>(r, at(j, true), S, j, live, dx, idx, sp);
      } else if (v * 32 + lane < nl) {
        const int j = list_l[v * 32 + lane];
        double x[M];
        limiter_line<double, DIR, true>(r, at(j, true), S, dx, idx, sp, x);
#pragma unroll
        for (int c = 0; c < M; ++c) r.lim(c, j) = x[c];
      }
    }
  }
}

// ---------------------------------------------------------------------------
// The wide form of the item phases, for launches that leave SMs idle: several
// threads per item share its work by roles, so that the phase takes the time
// of one role's instruction stream and every sub-partition has warps to
// interleave. Roles: the two sides of an interface (FIELDS: one per side and
// field), the limiter (FIELDS: one per field), the derivative flux and (LIN:
// scalar equations in 1D; else the same threads' second task) the linear part
// in FP64, each of whose chains of FP64 operations takes as long as a side.
// The
// arithmetic of every quantity is that of interface_line and limiter_line,
// operation for operation, so the results are the same bits.
// ---------------------------------------------------------------------------
template <int M, bool FIELDS, bool LIN = false>
struct WideRoles {
  static constexpr int sides = FIELDS ? 2 * M : 2, limiter = FIELDS ? M : 1;
  static constexpr int count = sides + limiter + 1 + LIN;
  // exchange rows of LI pairs: sides' fields, "-" side's linear parts, the
  // limiter's fields; then the bounds of the sides' and the limiter's fields
  static constexpr int rows = 7 * M;
};

// The lists of a tile's items for FP64.
template <int MAX>
struct ItemLists {
  int nf, nl;
  unsigned short f[MAX], l[MAX];
};

// Phases 3 and 3b for role `role` of interface j (left point kf) and point j
// (kl). xch: exchange rows. Every thread of the CTA calls it; C, D and lim
// are ready after the next barrier.
template <int DIR, bool FIELDS, bool LIN = false, class T, class L, class At>
__device__ __forceinline__ void wide_items(const T& r, D2* xch, int role, int j, bool has_f, int kf,
                                           bool has_l, int kl, int S, double alpha, double dx,
                                           double idx, const SchemeParams& sp, L& ls, At at,
                                           int rot) {
  constexpr int M = T::M;
  using R = WideRoles<M, FIELDS, LIN>;
  const LineData<D2, T> in(r, S, alpha, dx, sp);
  auto row = [&](int q) -> D2& { return xch[q * r.LI + j]; };
  CharOf<T, D2, DIR> ch;
  D2 f[M], lin[M];
  const int sd = FIELDS ? role / M : role, q0 = FIELDS ? role % M : 0;
  const bool lim_role = role >= R::sides && role < R::sides + R::limiter;
  const int lq = role - R::sides;
  const bool limited = sp.limiter != 0, chars = T::EUL && sp.limiter != 2;
  // items that are tried in pairs (every role of an item finds the same)
  const Route route = has_f ? interface_route(in, kf, S, alpha) : Route{false, true};
  const bool try_f = route.pairs;
  const bool try_l = FIELDS && lim_role && has_l && limited && limiter_fine(in, kl, S);
  if (role < R::sides) {
    if (try_f) {
      const LineWeights<D2> w = line_weights<D2>(sp, false);
      ch = char_system<DIR>(in, kf, true);
#pragma unroll
      for (int c = 0; c < M; ++c) f[c] = lin[c] = D2{0.f, 0.f};
      row(4 * M + sd * M + q0).h = interface_side<DIR, FIELDS>(in, ch, w, sd, kf, S, f, lin, q0);
      if constexpr (FIELDS) {
        row(sd * M + q0) = f[0];
      } else {
#pragma unroll
        for (int c = 0; c < M; ++c) row(sd * M + c) = f[c];
      }
      if (sd == 1 && q0 == 0)
#pragma unroll
        for (int c = 0; c < M; ++c) row(2 * M + c) = lin[c];
    }
  } else if (lim_role) {
    if (has_l && limited) {
      if constexpr (FIELDS) {
        float e = 0.f;
        if (try_l) row(3 * M + lq) = limiter_field<DIR>(in, ch, kl, S, sp, lq, e);
        row(6 * M + lq).h = e;
      } else {
        double x[M];
        if (!limiter_line<D2, DIR>(r, kl, S, dx, idx, sp, x))
          ls.l[atomicAdd(&ls.nl, 1)] = (unsigned short)j;
#pragma unroll
        for (int c = 0; c < M; ++c) r.lim(c, j) = x[c];
      }
    }
  } else if (role == R::sides + R::limiter && (T::EUL ? try_f : has_f)) {
#pragma unroll 1  // (code to fetch)
    for (int c = 0; c < M; ++c) {
      Q2 x[5];
      sides_differences(in, c, kf, S, x);
      r.D(c, j) = derivative_flux(in, x, c, kf, S, alpha, dx);
    }
  }
  if (role == R::count - 1 && try_f && !route.linear)
    r.C(0, j) = linear_part_fp64(r, kf, S, alpha, dx);
  __syncthreads();
  if (role == 0 && has_f && !try_f) ls.f[atomicAdd(&ls.nf, 1)] = (unsigned short)j;
  if (role == 0 && try_f) {
    double cc[M];
    float e[2] = {0.f, 0.f};
#pragma unroll
    for (int c = 0; c < M; ++c) {
      f[c] = add(row(c), row(M + c));
      lin[c] = add(lin[c], row(2 * M + c));
      if (FIELDS || c == 0) {  // (in the order of the loop over fields)
        e[0] += row(4 * M + c).h;
        e[1] += row(5 * M + c).h;
      }
    }
    interface_value<DIR>(in, ch, kf, S, alpha, f, lin, route.linear, r.C(0, j), cc);
    if (!interface_weak(r, kf, S, e[0] + e[1], alpha, sp))
      ls.f[atomicAdd(&ls.nf, 1)] = (unsigned short)j;
#pragma unroll
    for (int c = 0; c < M; ++c) r.C(c, j) = cc[c];
  }
  if constexpr (FIELDS) {
    if (lim_role && lq == 0 && has_l && limited && !try_l)
      ls.l[atomicAdd(&ls.nl, 1)] = (unsigned short)j;
    if (lim_role && lq == 0 && try_l) {
      D2 z[M];
      double x[M];
      float e = 0.f;
#pragma unroll
      for (int c = 0; c < M; ++c) {
        z[c] = row(3 * M + c);
        e += row(6 * M + c).h;
      }
      limiter_sum<DIR>(in, ch, kl, S, idx, chars, z, x);
      if (!limiter_weak(r, kl, e, sp)) ls.l[atomicAdd(&ls.nl, 1)] = (unsigned short)j;
#pragma unroll
      for (int c = 0; c < M; ++c) r.lim(c, j) = x[c];
    }
  }
  __syncthreads();
  if (ls.nf + ls.nl > 0)  // uniform
    listed_items<DIR>(r, ls.f, ls.nf, ls.l, ls.nl, at, S, rot, alpha, dx, idx, sp);
}

}  // namespace hweno
