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

namespace hweno {

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
  static constexpr size_t bytes(int L, int LI) {
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
  // split pairs of side sd (0: H^+, P; 1: H^-, M)
  __device__ __forceinline__ D2& H(int sd, int c, int k) const { return p(sd * M + c, k); }
  __device__ __forceinline__ D2& X(int sd, int c, int k) const { return p((2 + sd) * M + c, k); }
  __device__ __forceinline__ D2 dU(int c, int k) const {
    if constexpr (SLIM) return mul(sub(X(0, c, k), X(1, c, k)), ial);
    else return p(4 * M + c, k);
  }
  __device__ __forceinline__ D2 Nx(int c, int k) const {
    if constexpr (SLIM) return mul(sub(H(0, c, k), H(1, c, k)), ial);
    else return p(5 * M + c, k);
  }
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

// The pairs of point k from the derivative N and h = A N of its state:
// H^{+-} = dx (h +- alpha N) / 2 and dx N.
template <class T>
__device__ __forceinline__ void point_pairs(const T& r, int k, const double* N, const double* h,
                                            D2 alp, D2 dxp) {
#pragma unroll
  for (int c = 0; c < T::M; ++c) {
    const D2 nx = mul(dxp, to_pair(N[c])), x = mul(dxp, to_pair(h[c])), y = mul(alp, nx);
    if constexpr (!T::SLIM) r.p(5 * T::M + c, k) = nx;
    r.H(0, c, k) = scale(add(x, y), 0.5f);
    r.H(1, c, k) = scale(sub(x, y), 0.5f);
  }
}

// The eigen-system's inputs at point k from rho, 1/rho, E + p and the
// velocities along and across the line.
template <class T>
__device__ __forceinline__ void point_eigen(const T& r, int k, double rho, double ir, double Ep,
                                            double un, double ut) {
  const D2 rp = scale_pair(rho);
  const D2 up = to_pair(un), tp = T::M == 4 ? to_pair(ut) : D2{};
  const D2 H = mul(to_pair(Ep), to_pair(ir));
  r.E(0, k) = mul(rp, rsqrt2(rp));
  r.E(1, k) = up;
  r.E(2, k) = H;
  if constexpr (T::M == 4) r.E(3, k) = tp;
}

// The edge between points k and k + S.
template <class T>
__device__ __forceinline__ void edge_pairs(const T& r, int k, int S, D2 alp) {
  D2 dU[T::M];
#pragma unroll
  for (int c = 0; c < T::M; ++c) {
    dU[c] = to_pair(r.U(c, k + S) - r.U(c, k));
    if constexpr (!T::SLIM) r.p(4 * T::M + c, k) = dU[c];
  }
#pragma unroll
  for (int c = 0; c < T::M; ++c) {
    const D2 dF = T::EUL && c == 0 ? dU[T::kn] : to_pair(r.F(c, k + S) - r.F(c, k));
    const D2 au = mul(alp, dU[c]);
    r.X(0, c, k) = scale(add(dF, au), 0.5f);
    r.X(1, c, k) = scale(sub(dF, au), 0.5f);
  }
}

// The data of a line as X: pairs from the tile's pair rows, or doubles
// formed from its double rows.
template <class X, class T>
struct LineData;
template <class T>
struct LineData<D2, T> {
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
  // velocities and enthalpy at point k, or the Roe average of k and k + S
  __device__ __forceinline__ void state(int k, bool edge, D2& un, D2& ut, D2& H) const {
    if (!edge) {
      un = r.E(1, k);
      H = r.E(2, k);
      if constexpr (T::M == 4) ut = r.E(3, k);
      return;
    }
    const D2 sl = r.E(0, k), sr = r.E(0, k + S);
    const D2 is = div(D2{1.f, 0.f}, add(sl, sr));
    auto roe = [&](int e) { return mul(madd(sl, r.E(e, k), mul(sr, r.E(e, k + S))), is); };
    un = roe(1);
    H = roe(2);
    if constexpr (T::M == 4) ut = roe(3);
  }
};
template <class T>
struct LineData<double, T> {
  const T& r;
  int S;
  double alpha, dx;
  const SchemeParams& sp;
  __device__ __forceinline__ LineData(const T& r_, int S_, double al, double d,
                                      const SchemeParams& sp_)
      : r(r_), S(S_), alpha(al), dx(d), sp(sp_) {}
  __device__ __forceinline__ double H(int sd, int c, int k) const {
    return mul(0.5 * dx, madd(sd ? -alpha : alpha, r.N(c, k), r.h(c, k)));
  }
  __device__ __forceinline__ double X(int sd, int c, int k) const {
    return mul(0.5, madd(sd ? -alpha : alpha, dU(c, k), sub(r.F(c, k + S), r.F(c, k))));
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
  __device__ __forceinline__ void state(int k, bool edge, double& un, double& ut, double& H) const {
    constexpr int M = T::M;
    double a[M], b[M];
#pragma unroll
    for (int c = 0; c < M; ++c) {
      a[c] = r.U(c, k);
      b[c] = edge ? r.U(c, k + S) : 0.0;
    }
    if (!edge) {
      prim(a, un, ut, H);
    } else if (sp.eig_avg == 0) {  // Roe average
      double uL, tL = 0.0, HL, uR, tR = 0.0, HR;
      prim(a, uL, tL, HL);
      prim(b, uR, tR, HR);
      const double sl = mul(a[0], rsqrt_fp64(a[0])), sr = mul(b[0], rsqrt_fp64(b[0]));
      const double is = recip_fp64(add(sl, sr));
      auto roe = [&](double x, double y) { return mul(add(mul(sl, x), mul(sr, y)), is); };
      un = roe(uL, uR);
      ut = roe(tL, tR);
      H = roe(HL, HR);
    } else {  // arithmetic mean state
#pragma unroll
      for (int c = 0; c < M; ++c) a[c] = mul(0.5, add(a[c], b[c]));
      prim(a, un, ut, H);
    }
  }
};

// c ? a + y : a
template <class X>
__device__ __forceinline__ X add_if(bool c, X a, X y) {
  return add(a, pick2(c, y, X{}));
}

// The stencil differences of side sd of the interface between k and k + S,
// component c (the arguments of side_correction): the "+" side is about point
// k, the "-" side about k + S. The latter reverses the stencil and negates H;
// with M the difference of f^- along an edge, all five quantities are the "+"
// side's expressions in M and H^- times -1.
template <class X, class T>
__device__ __forceinline__ void side_differences(const LineData<X, T>& in, int sd, int c, int k,
                                                 int S, X* x) {
  using P2 = typename Num<X>::Scale;
  const P2 sg = sd ? P2(-1) : P2(1);
  const int k0 = sd ? k + S : k, km = sd ? k0 + S : k0 - S, kp = sd ? k : k0 + S;
  // the edges (k - S, k), (k, k + S) or (k + S, k + 2 S), (k, k + S)
  const X Hm = in.H(sd, c, km), H0 = in.H(sd, c, k0), Hp = in.H(sd, c, kp);
  x[0] = scale(sub(H0, in.X(sd, c, sd ? k0 : km)), sg);
  x[1] = scale(sub(H0, in.X(sd, c, k)), sg);
  x[2] = scale(sub(add(Hm, Hp), scale(H0, P2(2))), sg);
  x[3] = scale(sub(Hm, Hp), sg);
  x[4] = scale(H0, sg);
}

// c of the interface between points k and k + S; in pairs, false when the
// correction is not small (the values are then not to be used).
template <class X, int DIR, class T>
__device__ __forceinline__ bool interface_line(const T& r, int k, int S, double alpha, double dx,
                                               const SchemeParams& sp, double* cc) {
  constexpr int M = T::M;
  constexpr bool FP64 = std::is_same<X, double>::value;
  const LineData<X, T> in(r, S, alpha, dx, sp);
  const LineWeights<X> w = line_weights<X>(sp, false);
  bool weak = true;
  LineChar<X, M == 1 ? 3 : M, M == 1 ? 0 : DIR> ch;
  if constexpr (T::EUL) {
    X un, ut{}, H;
    in.state(k, true, un, ut, H);
    const X q = ch.kinetic(un, ut);
    ch.init(un, ut, H, q, mul(in.gm1(), sub(H, q)), in.gm1());
  }
  auto side = [&](X y1, X y2, X s, X d, X H0) {
    if constexpr (FP64) return side_value(y1, y2, s, d, H0, w);
    else return side_correction(y1, y2, s, d, H0, w, weak);
  };
  X f[M], lin[M];
#pragma unroll
  for (int c = 0; c < M; ++c) f[c] = lin[c] = X{};
#pragma unroll 1
  for (int sd = 0; sd < 2; ++sd) {
    X x[M][5];
#pragma unroll
    for (int c = 0; c < M; ++c) {
      side_differences(in, sd, c, k, S, x[c]);
      if constexpr (!FP64) lin[c] = add(lin[c], linear_part(x[c][0], x[c][1], x[c][3]));
    }
    if constexpr (T::EUL) {
      typename decltype(ch)::Factors a[5];
#pragma unroll
      for (int v = 0; v < 5; ++v) {
        X y[M];
#pragma unroll
        for (int c = 0; c < M; ++c) y[c] = x[c][v];
        a[v] = ch.factors(y);
      }
#pragma unroll 1
      for (int q = 0; q < M; ++q) {
        const X y = side(a[0].field(q), a[1].field(q), a[2].field(q), a[3].field(q), a[4].field(q));
#pragma unroll
        for (int c = 0; c < M; ++c) f[c] = add_if(q == c, f[c], y);
      }
    } else {
      f[0] = add(f[0], side(x[0][0], x[0][1], x[0][2], x[0][3], x[0][4]));
    }
  }
  if constexpr (T::EUL) {
    X out[M];
    ch.right(f, out);
#pragma unroll
    for (int c = 0; c < M; ++c) f[c] = out[c];
  }
#pragma unroll
  for (int c = 0; c < M; ++c) {
    // f^+_i + f^-_{i+1} = (F_i + F_{i+1}) / 2 - alpha (U_{i+1} - U_i) / 2
    if constexpr (FP64) cc[c] = madd(-0.5 * alpha, in.dU(c, k), f[c]);
    else cc[c] = to_double(madd(dconst(1.0 / 60.0), lin[c], mul(f[c], dconst(1.0 / 12.0))));
  }
  return weak;
}

// The derivative flux dx (h-hat^+ + h-hat^-) of component c at the interface
// between k and k + S: both sides' p_0' of Sec. 2.1 in terms of F, U, h, N.
template <class T>
__device__ __forceinline__ double derivative_flux_fp64(const T& r, int c, int k, int S, double kU,
                                                       double kh, double kv) {
  const int m = k - S, p = k + S, q = k + 2 * S;
  const double t0 = r.F(c, p) - r.F(c, k), t1 = r.F(c, q) - r.F(c, m);
  const double su = (r.U(c, q) - r.U(c, p)) - (r.U(c, k) - r.U(c, m));
  const double sh = fma(-7.0, r.h(c, k) + r.h(c, p), r.h(c, m) + r.h(c, q));
  const double sv = fma(3.0, r.N(c, k) - r.N(c, p), r.N(c, m) - r.N(c, q));
  return fma(1.875, t0, fma(-0.125, t1, fma(kU, su, fma(kh, sh, kv * sv))));
}

// The limited derivative at point k; in pairs, false as interface_line.
template <class X, int DIR, class T>
__device__ __forceinline__ bool limiter_line(const T& r, int k, int S, double dx, double idx,
                                             const SchemeParams& sp, double* vt) {
  constexpr int M = T::M;
  const LineData<X, T> in(r, S, 0.0, dx, sp);
  bool weak = true;
  X x[4][M], z[M];
#pragma unroll
  for (int c = 0; c < M; ++c) {
    x[0][c] = in.dU(c, k - S);
    x[1][c] = in.dU(c, k);
    x[2][c] = in.Nx(c, k - S);
    x[3][c] = in.Nx(c, k + S);
  }
  const LineWeights<X> w = line_weights<X>(sp, true);
  auto limit = [&](X q1, X q2, X Vm, X Vp) {
    if constexpr (std::is_same<X, double>::value) return limiter_value(q1, q2, Vm, Vp, w);
    else return limiter_correction(q1, q2, Vm, Vp, w, weak);
  };
  if (T::EUL && sp.limiter != 2) {  // uniform
    if constexpr (T::EUL) {
      LineChar<X, M, DIR> ch;
      X un, ut{}, H, f[M];
      in.state(k, false, un, ut, H);
      const X q = ch.kinetic(un, ut);
      ch.init(un, ut, H, q, mul(in.gm1(), sub(H, q)), in.gm1());
      typename decltype(ch)::Factors a[4];
#pragma unroll
      for (int v = 0; v < 4; ++v) a[v] = ch.factors(x[v]);
#pragma unroll
      for (int c = 0; c < M; ++c) f[c] = X{};
#pragma unroll 1
      for (int q = 0; q < M; ++q) {
        const X y = limit(a[0].field(q), a[1].field(q), a[2].field(q), a[3].field(q));
#pragma unroll
        for (int c = 0; c < M; ++c) f[c] = pick2(q == c, y, f[c]);
      }
      ch.right(f, z);
    }
  } else {
#pragma unroll
    for (int c = 0; c < M; ++c) z[c] = limit(x[0][c], x[1][c], x[2][c], x[3][c]);
  }
  // dx q_0' = 3/4 (u_{i+1} - u_{i-1}) - dx (v_{i-1} + v_{i+1}) / 4
  const double k3 = 0.75 * idx, k1 = 0.25 * idx;
#pragma unroll
  for (int c = 0; c < M; ++c) {
    if constexpr (std::is_same<X, double>::value) {
      vt[c] = mul(idx, z[c]);
    } else {
      const double q0 =
          fma(k3, r.U(c, k + S) - r.U(c, k - S), -0.25 * (r.N(c, k - S) + r.N(c, k + S)));
      vt[c] = fma(k1, to_double(z[c].l), fma(k1, to_double(z[c].h), q0));
    }
  }
  return weak;
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
    double a[M], un, ut = 0.0, H;
    if (sp.eig_avg == 0) {  // Roe average; each side's lanes take one state
#pragma unroll
      for (int i = 0; i < M; ++i) a[i] = r.U(i, sd ? k + S : k);
      in.prim(a, un, ut, H);
      const double s = mul(a[0], rsqrt_fp64(a[0]));
      const double so = __shfl_xor_sync(all, s, NC), is = recip_fp64(add(s, so));
      auto roe = [&](double x) {
        const double m = mul(s, x), o = __shfl_xor_sync(all, m, NC);
        return mul(add(m, o), is);
      };
      un = roe(un);
      H = roe(H);
      if constexpr (M == 4) ut = roe(ut);
    } else {
#pragma unroll
      for (int i = 0; i < M; ++i) a[i] = mul(0.5, add(r.U(i, k), r.U(i, k + S)));
      in.prim(a, un, ut, H);
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
      LineChar<double, M, DIR> ch;
      double un, ut = 0.0, H;
      in.state(k, false, un, ut, H);
      const double kin = ch.kinetic(un, ut);
      ch.init(un, ut, H, kin, mul(in.gm1(), sub(H, kin)), in.gm1());
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
  // groups: 150 instructions per 32 / kInterface interfaces and warp; whole
  // items: 450 per 32 (limiter: 115 and 300)
  constexpr int gf = 32 / G::kInterface, gl = 32 / G::kPoint;
  const bool few_f = nf <= 3 * gf * nw, few_l = nl <= 3 * gl * nw;
  const int uf = few_f ? (nf + gf - 1) / gf : (nf + 31) / 32;
  const int ul = few_l ? (nl + gl - 1) / gl : (nl + 31) / 32;
  for (int u = (warp + rot) % nw; u < uf + ul; u += nw) {
    if (u < uf) {
      if (few_f) {
        const int i = u * gf + lane / G::kInterface;
        const bool live = i < nf;
        const int j = list_f[live ? i : 0];
        interface_group<DIR>(r, at(j, false), S, j, live, alpha, dx, sp);
      } else if (u * 32 + lane < nf) {
        const int j = list_f[u * 32 + lane];
        double x[M];
        interface_line<double, DIR>(r, at(j, false), S, alpha, dx, sp, x);
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
        limiter_line<double, DIR>(r, at(j, true), S, dx, idx, sp, x);
#pragma unroll
        for (int c = 0; c < M; ++c) r.lim(c, j) = x[c];
      }
    }
  }
}

}  // namespace hweno
