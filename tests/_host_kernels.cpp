// Device functions of the FP64 kernels compiled for the host (_host_cuda.h),
// for tests that need no GPU.
#include "_host_cuda.h"

#include "hweno.h"
#include "flux2d.cuh"
#include "hweno_adjoint.cuh"
#include "internal.h"
#include "line_df.cuh"
#include "rough_speed.cuh"
#include "stage2d_common.cuh"

using namespace hweno;

namespace {

struct Opts {
  double g[3], d[3], eps, gamma;
  int limiter, eig_avg;
};

SchemeParams params(const Opts& o) {
  SchemeParams sp{};
  fill_constant_table(sp, o.g, o.d, o.eps, o.gamma, 0.0);
  sp.limiter = o.limiter;
  sp.eig_avg = o.eig_avg;
  return sp;
}

// One point of a periodic line: state u, derivative v, flux F, h = f'(u) v and
// (Euler) 1/rho, E + p and the velocities.
template <int M>
struct Point {
  double u[M], v[M], F[M], h[M], ir = 0, Ep = 0, un = 0, ut = 0, p = 0;
  Point(int eq, int n, int s, const double* U, const double* V, double gm1) {
    for (int c = 0; c < M; ++c) {
      u[c] = U[c * n + s];
      v[c] = V[c * n + s];
    }
    if (eq == HWENO_BURGERS) {
      F[0] = 0.5 * u[0] * u[0];
      h[0] = u[0] * v[0];
    } else if (eq == HWENO_BUCKLEY) {
      const double w = 1.0 - u[0], iD = recip_fp64(std::fma(w, w, 4.0 * u[0] * u[0]));
      F[0] = 4.0 * u[0] * u[0] * iD;
      h[0] = 8.0 * u[0] * w * (iD * iD) * v[0];
    } else {
      double a[4] = {u[0], u[1], M == 4 ? u[2] : 0.0, u[M - 1]}, f[4], b[4] = {v[0], v[1], 0.0, 0.0};
      b[2] = M == 4 ? v[2] : 0.0;
      b[3] = v[M - 1];
      const Prim2<double> q = prim2_ir(a, gm1, recip_fp64(u[0]));
      double k[4];
      flux2<HWENO_EULER, 0>(a, q, f);
      jvp2<HWENO_EULER, 0>(a, q, b, gm1, k);
      for (int c = 0; c < M; ++c) {
        F[c] = f[c == M - 1 ? 3 : c];
        h[c] = k[c == M - 1 ? 3 : c];
      }
      ir = q.ir;
      Ep = q.Ep;
      un = q.u;
      ut = q.v;
      p = q.p;
    }
  }
};

// L^1, L^2 and v~ of a periodic line by the FP64 kernels' phases
// (stage1d_df.cuh, stage2d_df.cuh) on one tile; listed[0], listed[1]: the
// interfaces and points evaluated in FP64.
template <int M, bool EUL, bool SLIM>
void line_pairs(int eq, int n, double dx, double alpha, const double* U, const double* V,
                const Opts& o, double* L1, double* L2, double* Vt, int* listed) {
  using T = LineTile<M, 0, EUL, 0, SLIM>;
  const SchemeParams sp = params(o);
  const int L = n + 4, LI = n + 1;
  std::vector<double> mem(T::bytes(L, LI) / sizeof(double) + 1);
  unsigned status = 0;
  const D2 alp = scale_pair(alpha), dxp = to_pair(dx);
  const T r{mem.data(), L, LI, &status, SLIM ? div(D2{1.f, 0.f}, alp) : D2{}};
  const double idx = 1.0 / dx;
  for (int g = 0; g < L; ++g) {
    const Point<M> q(eq, n, (g - 2 + n) % n, U, V, o.gamma - 1.0);
    for (int c = 0; c < M; ++c) {
      r.U(c, g) = q.u[c];
      r.N(c, g) = q.v[c];
      if (!EUL || c > 0) {
        r.F(c, g) = q.F[c];
        r.h(c, g) = q.h[c];
      }
    }
    if constexpr (EUL) point_eigen(r, g, q.u[0], q.ir, q.Ep, q.un, q.ut);
    point_pairs(r, g, q.v, q.h, alp, dxp);
  }
  for (int g = 0; g < L - 1; ++g) edge_pairs(r, g, 1, alp);
  for (int j = 0; j <= n; ++j) {
    double x[M], d[M];
    if (!interface_line<D2, 0>(r, j + 1, 1, alpha, dx, sp, x, d)) {
      listed[0] += j < n;
      interface_line<double, 0>(r, j + 1, 1, alpha, dx, sp, x);
      if (EUL)
        for (int c = 0; c < M; ++c) d[c] = derivative_flux_fp64(r, c, j + 1, 1, alpha, dx);
    }
    for (int c = 0; c < M; ++c) {
      r.C(c, j) = x[c];
      r.D(c, j) = d[c];
    }
    if (j == n) break;
    if (!limiter_line<D2, 0>(r, j + 2, 1, dx, idx, sp, x)) {
      ++listed[1];
      limiter_line<double, 0>(r, j + 2, 1, dx, idx, sp, x);
    }
    for (int c = 0; c < M; ++c) r.lim(c, j) = x[c];
  }
  for (int c = 0; c < M; ++c)
    for (int j = 0; j < n; ++j) {
      const int g = j + 2, q = c * n + j;
      const double dF =
          std::fma(0.5, r.F(c, g + 1) - r.F(c, g - 1), r.C(c, j + 1) - r.C(c, j));
      L1[q] = -dF * idx;
      L2[q] = -(r.D(c, j + 1) - r.D(c, j)) * (idx * idx);
      Vt[q] = r.lim(c, j);
    }
}

// The same by the all-FP64 form (hweno_math.cuh, the kernels that keep it).
template <int M, bool EUL>
void line_fp64(int eq, int n, double dx, double alpha, const double* U, const double* V,
               const Opts& o, double* L1, double* L2, double* Vt) {
  const SchemeParams sp = params(o);
  const Weights<double> w = weights_from(sp.wd);
  const double gm1 = o.gamma - 1.0, idx = 1.0 / dx;
  const int L = n + 4;
  std::vector<Point<M>> P;
  std::vector<double> s[6][M], F[M], D[M];
  for (auto& a : s)
    for (auto& b : a) b.resize(L);
  for (auto& a : F) a.resize(n + 1);
  for (auto& a : D) a.resize(n + 1);
  for (int g = 0; g < L; ++g) {
    P.emplace_back(eq, n, (g - 2 + n) % n, U, V, gm1);
    for (int c = 0; c < M; ++c) {
      s[0][c][g] = P[g].u[c];
      s[1][c][g] = dx * P[g].v[c];
      split_pm(P[g].F[c], P[g].u[c], P[g].h[c], P[g].v[c], 0.5 * alpha, 0.5 * dx * alpha, 0.5 * dx,
               s[2][c][g], s[3][c][g], s[4][c][g], s[5][c][g]);
    }
  }
  auto system = [&](double un, double ut, double H) {
    Char2<double, 0> ch;
    ch.init(un, ut, H, gm1 * (H - 0.5 * (un * un + ut * ut)), gm1);
    return ch;
  };
  // row q of the system's left matrix applied to array k at point g
  auto left = [&](const Char2<double, 0>& ch, int q, int k, int g) {
    return ch.left(M == 3 && q == 2 ? 3 : q, s[k][0][g], s[k][M > 1 ? 1 : 0][g],
                   M == 4 ? s[k][2 % M][g] : 0.0, s[k][M - 1][g]);
  };
  auto right = [&](const Char2<double, 0>& ch, const double* z, double* out) {
    const double a[4] = {z[0], z[1], M == 4 ? z[2] : 0.0, z[M - 1]};
    double b[4];
    ch.right(a, b);
    for (int c = 0; c < M; ++c) out[c] = b[c == M - 1 ? 3 : c];
  };
  for (int j = 0; j <= n; ++j) {
    const int g = j + 1;
    double z[4], f[4];
    Char2<double, 0> ch;
    if (EUL) {
      // the Roe average, or the arithmetic mean state
      const double a = std::sqrt(P[g].u[0]), b = std::sqrt(P[g + 1].u[0]), is = 1.0 / (a + b);
      auto roe = [&](double x, double y) { return (a * x + b * y) * is; };
      ch = system(roe(P[g].un, P[g + 1].un), roe(P[g].ut, P[g + 1].ut),
                  roe(P[g].Ep * P[g].ir, P[g + 1].Ep * P[g + 1].ir));
      if (o.eig_avg) {
        auto mean = [&](int c) { return 0.5 * (P[g].u[c] + P[g + 1].u[c]); };
        const double ir = 1.0 / mean(0), un = mean(1) * ir, ut = M == 4 ? mean(2 % M) * ir : 0.0;
        const double kin = 0.5 * (mean(1) * un + (M == 4 ? mean(2 % M) * ut : 0.0));
        ch = system(un, ut, (mean(M - 1) + gm1 * (mean(M - 1) - kin)) * ir);
      }
    }
    for (int q = 0; q < M; ++q) {
      auto x = [&](int k, int i) { return EUL ? left(ch, q, k, i) : s[k][q][i]; };
      z[q] = interface_flux(x(2, g - 1), x(2, g), x(2, g + 1), x(4, g - 1), x(4, g), x(4, g + 1),
                            x(3, g), x(3, g + 1), x(3, g + 2), x(5, g), x(5, g + 1), x(5, g + 2), w);
    }
    if (EUL) right(ch, z, f);
    for (int c = 0; c < M; ++c) {
      F[c][j] = EUL ? f[c] : z[c];
      const auto &a = s[2][c], &b = s[3][c], &p = s[4][c], &m = s[5][c];
      D[c][j] = derivative_flux(a[g - 1], a[g], a[g + 1], p[g - 1], p[g], p[g + 1], b[g], b[g + 1],
                                b[g + 2], m[g], m[g + 1], m[g + 2]);
    }
  }
  for (int j = 0; j < n; ++j) {
    const int g = j + 2;
    const bool chars = EUL && o.limiter != 2;
    Char2<double, 0> ch;
    double z[4], out[4];
    if (chars) ch = system(P[g].un, P[g].ut, P[g].Ep * P[g].ir);
    for (int q = 0; q < M; ++q) {
      auto x = [&](int k, int i) { return chars ? left(ch, q, k, i) : s[k][q][i]; };
      z[q] = limited_derivative(x(0, g - 1), x(0, g), x(0, g + 1), x(1, g - 1), x(1, g + 1), w);
    }
    if (chars) right(ch, z, out);
    for (int c = 0; c < M; ++c) {
      L1[c * n + j] = -(F[c][j + 1] - F[c][j]) * idx;
      L2[c * n + j] = -(D[c][j + 1] - D[c][j]) * (idx * idx);
      Vt[c * n + j] = (chars ? out[c] : z[c]) * idx;
    }
  }
}

}  // namespace

extern "C" {

// n states u[i][4] (M used): the FP32 speeds of direction x (and, 2D, y)
void host_rough_speeds(int eq, int dim, int n, const double* u, double gamma, float* sx,
                       float* sy) {
  for (int i = 0; i < n; ++i, u += 4) {
    const float g = (float)gamma;
    if (dim == 2) {
      if (eq == HWENO_EULER) rough_speeds2<HWENO_EULER>(u, g, sx[i], sy[i]);
      else rough_speeds2<HWENO_BURGERS>(u, g, sx[i], sy[i]);
    } else {
      sx[i] = eq == HWENO_EULER     ? rough_speed<HWENO_EULER>(u, g)
              : eq == HWENO_BUCKLEY ? rough_speed<HWENO_BUCKLEY>(u, g)
                                    : rough_speed<HWENO_BURGERS>(u, g);
    }
  }
}

// side_vjp (limiter = 0) or limiter_vjp of n stencils x[i][6] (5 used by the
// limiter) with cotangent 1: values v[i] and gradients g[i][6]
void host_vjp(int limiter, int n, const double* x, const double* w3, double eps, double* v,
              double* g) {
  Weights<double> w{};
  w.g0 = w.d0 = w3[0];
  w.g1 = w.d1 = w3[1];
  w.g2 = w.d2 = w3[2];
  w.eps = eps;
  for (int i = 0; i < n; ++i, x += 6, g += 6) {
    for (int k = 0; k < 6; ++k) g[k] = 0.0;
    v[i] = limiter ? limiter_vjp(x[0], x[1], x[2], x[3], x[4], 1.0, w, g)
                   : side_vjp(x[0], x[1], x[2], x[3], x[4], x[5], 1.0, w, g);
  }
}

// L^1, L^2, v~ of a periodic line of n points, m components: by the pair
// kernels' functions (form 0: 1D tiles, 1: 2D tiles) or the all-FP64 form (2)
void host_line(int form, int eq, int m, int n, double dx, double alpha, const double* U,
               const double* V, const double* lin_w, const double* lim_d, double eps, double gamma,
               int limiter, int eig_avg, double* L1, double* L2, double* Vt, int* listed) {
  const Opts o{{lin_w[0], lin_w[1], lin_w[2]}, {lim_d[0], lim_d[1], lim_d[2]}, eps, gamma, limiter,
               eig_avg};
  if (form == 2) {
    auto* f = m == 1 ? line_fp64<1, false> : m == 3 ? line_fp64<3, true> : line_fp64<4, true>;
    return f(eq, n, dx, alpha, U, V, o, L1, L2, Vt);
  }
  auto* f = m == 1   ? (form ? line_pairs<1, false, true> : line_pairs<1, false, false>)
            : m == 3 ? line_pairs<3, true, false>
                     : line_pairs<4, true, true>;
  f(eq, n, dx, alpha, U, V, o, L1, L2, Vt, listed);
}

// Arithmetic of dfloat.cuh and weno_df.cuh: operation `op` on a[i] and b[i]
// (pairs made by to_pair, but those of op 4), results r[i] and, pairs, both words
void host_arith(int op, int n, const double* a, const double* b, double* r, float* h, float* l) {
  for (int i = 0; i < n; ++i) {
    D2 x = to_pair(a[i]);
    const D2 y = to_pair(b[i]);
    switch (op) {
      case 0: break;
      case 1: x = div(x, y); break;
      case 2: x = rsqrt2(x); break;
      case 3: x = mul(x, y); break;
      case 4: x = D2{(float)a[i], (float)b[i]}; break;
      case 5: x = madd(x, y, D2{1.f, 0.f}); break;
      case 6: x = add(x, y); break;
    }
    h[i] = x.h;
    l[i] = x.l;
    r[i] = op == 4 ? to_double(x.h) : op == 7 ? recip_fp64(a[i])
           : op == 8 ? rsqrt_fp64(a[i]) : op == 9 ? (double)to_float(a[i]) : to_double(x);
  }
}
// whether n listed items go to groups of lanes (interfaces, limiter points)
int host_few(int m, int limiter, int n) {
  using A = LineTile<1, 0, false>;
  using B = LineTile<3, 0, true>;
  auto few = [&](auto g) {
    using G = decltype(g);
    return limiter ? G::few(n, G::kPoint, G::group_l, G::whole_l)
                   : G::few(n, G::kInterface, G::group_f, G::whole_f);
  };
  return m == 1 ? few(Group<A>{}) : few(Group<B>{});
}
}
