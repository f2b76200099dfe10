// Reverse-mode derivatives (vector-Jacobian products) of the scalar building
// blocks of the L-HWENO stage (Zhang & Zhao, arXiv:2207.05258, Sec. 2.1-2.2),
// written by hand from a form in the differences of the stencil: the
// indicators as sums of squares of triangular factorisations (weno_df.cuh),
// the weights over their common denominator. Equal in exact arithmetic to the
// paper's form, with one reciprocal and no division. The FP64 pipe bounds
// these kernels: about 100 operations a side, where the per-weight form in
// full values took 61 + 75 and 11 divisions (256 x 256 density wave, one step's
// adjoint, FP64: 5.19 -> 4.20 ms; batch of Burgers gradients 9.38 -> 7.33 ms).
// Root-mean-square error of a side's gradient against long double, per-weight
// form -> this one, on smooth data / next to a jump / on noise: 2.1e-17 /
// 2.9e-14 / 7.8e-16 -> 2.1e-17 / 3.2e-17 / 4.8e-17; of the limiter's: 5.4e-17 /
// 1.9e-16 / 2.8e-16 -> 2.6e-17 / 5.1e-17 / 2.2e-16; of the values: 0.3 to 0.98
// of the per-weight form's. The |.| in tau keeps the sign of
// its argument at the point of evaluation (the branch of the forward run).
// With `frozen` the nonlinear weights count as constants: only the
// candidates' (linear) dependence on the data is propagated.
#pragma once

#include "hweno_math.cuh"
#include "weno_df.cuh"

namespace hweno {

namespace adj {
// coefficients of flux_indicators and limiter_indicators
constexpr double F1 = 9883630.0 / 3288933.0, F2 = 44358.0 / 22025.0;
constexpr double FZ1 = 1096311.0 / 1120.0, FG = 21520059541.0 / 2210162976.0;
constexpr double FZ2 = 4405.0 / 112.0, FL = 1421461.0 / 1321500.0, FY = 13.0 / 3.0;
constexpr double L1 = -120.0 / 3169.0, L2 = 527690.0 / 262907.0;
constexpr double LZ1 = 3169.0 / 1280.0, LU = 781.0 / 3169.0;
constexpr double LZ2 = 262907.0 / 6720.0, LL = 1421461.0 / 1314535.0;
// beta_0 of the reconstruction as H_i^2 + E2^2 + E3^2 + A4^2 + K11 a5^2, E2 =
// E2d d + E2l lap, E3 = E3s s + E3d g, A4 = A4d d + A4l lap, a5 = s/4 + 3/4 g
// (square roots times the exact coefficients, to 20 digits; E3h: E3's
// coefficient of H_i over s + 2 H_i and g - 2 H_i). The factorised
// coefficients above are those of the same quadratic form.
constexpr double K11 = 21520059541.0 / 1377684.0;
constexpr double E2d = 0.52842290755678754049, E2l = 2.0976788148466414486;
constexpr double E3s = -1.6032089149031235916, E3h = -12.661835579599691806,
                 E3d = -7.9341267047029694945;
constexpr double A4d = -6.2490900436484649542, A4l = -12.498180087296929908;
constexpr bool same(double x, double y) { return x - y < 1e-10 && y - x < 1e-10; }
static_assert(same(2.0 * E3s + E3h, 2.0 * E3d), "E3 is free of H_i");
static_assert(same(FZ1, E3s * E3s + K11 / 16.0), "s s");
static_assert(same(FZ1 * F1, E3s * E3d + K11 * 3.0 / 16.0), "s g");
static_assert(same(FZ1 * F1 * F1 + FG, E3d * E3d + K11 * 9.0 / 16.0), "g g");
static_assert(same(FZ2, E2d * E2d + A4d * A4d), "d d");
static_assert(same(FZ2 * F2, E2d * E2l + A4d * A4l), "d lap");
static_assert(same(FZ2 * F2 * F2 + FL, E2l * E2l + A4l * A4l), "lap lap");
}  // namespace adj

// Source of point p of an instance with n points (maybe a ghost): kind 0
// copy, 1 mirror (reflective wall), 2 imposed state (no dependence on the
// instance's values). Same mapping as the forward stage's loads.
__device__ __forceinline__ int ghost_src(int p, int n, int bclo, int bchi, int& kind) {
  kind = 0;
  if (p >= 0 && p < n) return p;
  const int b = p < 0 ? bclo : bchi;
  if (b == HWENO_BC_PERIODIC) return p < 0 ? p + n : p - n;
  if (b == HWENO_BC_OUTFLOW) return p < 0 ? 0 : n - 1;
  if (b == HWENO_BC_REFLECTIVE) { kind = 1; return p < 0 ? -p - 1 : 2 * n - 1 - p; }
  kind = 2;
  return 0;
}

// x with the sign of y; 0 where y is 0.
__device__ __forceinline__ double signed_by(double x, double y) {
  const int flip = __double2hiint(y) & (int)0x80000000;
  const double r = __hiloint2double(__double2hiint(x) ^ flip, __double2loint(x));
  const bool zero = ((__double2hiint(y) & 0x7fffffff) | __double2loint(y)) == 0;
  return zero ? 0.0 : r;
}

// The nonlinear value v = sum of phi_l p_l of weno_df.cuh, with phi_0 =
// b_1 b_2 (b_0 + tau) / D, phi_l = tau n_l / D, n_l = q_l (b_0 - b_l),
// q_1 = g_1 b_2, q_2 = g_2 b_1, from the indicators b_l (eps included), p_l,
// P_l = p_l - p_0, P = p_1 - p_2 and the linear weights (their sum is 1);
// gp_l = mu phi_l and, unless `frozen`, gb_l = mu dv / d b_l (tau's included).
// The latter in r_l = p_l - v, formed from the differences and the phi: small
// where p_l has most of the weight, accurate where all differences are small.
__device__ __forceinline__ double weighted_vjp(double b0, double b1, double b2, double p0,
                                               double p1, double p2, double P1, double P2,
                                               double P, double g0, double g1, double g2,
                                               double mu, bool frozen, double& gp0, double& gp1,
                                               double& gp2, double& gb0, double& gb1,
                                               double& gb2) {
  // The denominator is of degree four in the indicators (tau of degree two).
  // From 2^240 on they are scaled by the power of two of b_0 (the others
  // exceed it by at most 2%), tau, of which the weights take tau / b, by the
  // same, and the cotangents of the b_l back: finite up to indicators of about
  // 1e260. By integer operations on the exponents (a branch around FP64 ones
  // cost 2% of the 2D adjoint); with sh = 0 nothing changes.
  const int ex = __double2hiint(b0) & 0x7ff00000;
  const int sh = ex > (1023 + 240) << 20 && ex != 0x7ff00000 ? ex - (1023 << 20) : 0;
  auto shift = [](double x, int by) {  // x 2^by; 0 or less where it underflows
    return __hiloint2double(max(__double2hiint(x) + by, 0), __double2loint(x));
  };
  b0 = shift(b0, -sh);
  b1 = shift(b1, -sh);
  b2 = shift(b2, -sh);
  const double e1 = b0 - b1, e2 = b0 - b2;
  const double ht = 0.5 * (fabs(e1) + fabs(e2)), tau = shift(ht * ht, sh);
  const double q1 = g1 * b2, q2 = g2 * b1, n1 = q1 * e1, n2 = q2 * e2;
  const double b12 = b1 * b2, bt = b0 + tau;
  const double iD = recip_fp64(b12 * (b0 + g0 * tau) + tau * (b0 * (q1 + q2)));
  const double tD = tau * iD;
  double f0 = b12 * bt * iD, f1 = tD * n1, f2 = tD * n2;
  // the largest weight by the other two, whose errors are smaller: phi_0 from 1/2
  // on, the others from 15/16
  const bool m0 = __double2hiint(f0) >= 0x3fe00000, m1 = __double2hiint(f1) >= 0x3fee0000;
  const bool m2 = __double2hiint(f2) >= 0x3fee0000;
  const double most = 1.0 - ((m0 ? f1 : f0) + (m2 ? f1 : f2));
  if (m0) f0 = most;
  else if (m1) f1 = most;
  else if (m2) f2 = most;
  const double r0 = -(f1 * P1 + f2 * P2);
  gp0 = mu * f0;
  gp1 = mu * f1;
  gp2 = mu * f2;
  gb0 = gb1 = gb2 = 0.0;
  if (!frozen) {
    const double m = mu * iD, mt = m * tau;
    const double r1 = f0 * P1 + f2 * P, r2 = f0 * P2 - f1 * P, x = r0 * b12;
    const double gt = ht * m * (x + (r1 * n1 + r2 * n2));  // t / 2 times the cotangent of tau
    const double t1 = signed_by(gt, e1), t2 = signed_by(gt, e2);
    const double k = m * bt * r0 - mt * (g1 * r1 + g2 * r2), mb = mt * b0;
    // (in gt the powers of tau and of the b_l cancel)
    const double down = __hiloint2double((1023 << 20) - sh, 0);
    gb0 = (m * x + mt * (r1 * q1 + r2 * q2)) * down + (t1 + t2);
    gb1 = (b2 * k + g2 * (mb * r2)) * down - t1;
    gb2 = (b1 * k + g1 * (mb * r1)) * down - t2;
  }
  return f0 * p0 + (f1 * p1 + f2 * p2);
}

// One side of the nonlinear flux, f-hat^+ from (f, H = dx h) on {i-1, i, i+1}
// (Sec. 2.1): returns the value and adds mu * d f-hat / d input to g[6]
// (order fm, f0, fp, Hm, H0, Hp).
__device__ __forceinline__ double side_vjp(double fm, double f0, double fp, double Hm, double H0,
                                           double Hp, double mu, const Weights<double>& w,
                                           double* g, bool frozen = false) {
  using namespace adj;
  const double y1 = (fm - f0) + H0, y2 = (f0 - fp) + H0, s = (Hm + Hp) - 2.0 * H0, d = Hm - Hp;
  const double gg = y1 + y2, lap = y1 - y2;
  const double z1 = s + F1 * gg, z2 = d + F2 * lap;
  const double c1 = FZ1 * z1, cg = FG * gg, c2 = FZ2 * z2, cl = FL * lap;
  const double k1 = FY * y1, k2 = FY * y2, h = H0 * H0 + w.eps;
  const double b0 = c1 * z1 + (cg * gg + (c2 * z2 + (cl * lap + h)));
  // p_l relative to f0; 60 P_l = +-5 g - 3 (d + 2 lap)
  const double h0 = 0.5 * H0, p0 = 11.0 / 60.0 * lap + (0.05 * d + h0);
  const double c = 0.05 * (d + 2.0 * lap), e = 1.0 / 12.0 * gg;
  double gp0, gp1, gp2, gb0, gb1, gb2;
  const double v = weighted_vjp(b0, k1 * y1 + h, k2 * y2 + h, p0, 1.0 / 6.0 * y1 + h0,
                                h0 - 1.0 / 6.0 * y2, e - c, -e - c, 2.0 * e, w.g0, w.g1, w.g2, mu,
                                frozen, gp0, gp1, gp2, gb0, gb1, gb2);
  const double t0 = 2.0 * gb0;
  const double gs = t0 * c1, gz2 = t0 * c2, gdd = gz2 + 0.05 * gp0;
  const double ggg = F1 * gs + t0 * cg, gl = F2 * gz2 + (t0 * cl + 11.0 / 60.0 * gp0);
  const double gy1 = 2.0 * (gb1 * k1) + (1.0 / 6.0 * gp1 + (ggg + gl));
  const double gy2 = 2.0 * (gb2 * k2) - (1.0 / 6.0 * gp2 - (ggg - gl));
  g[0] += gy1;
  g[1] += mu - (gy1 - gy2);
  g[2] -= gy2;
  g[3] += gs + gdd;
  g[4] += 0.5 * mu + 2.0 * (H0 * (gb0 + (gb1 + gb2)) - gs) + (gy1 + gy2);
  g[5] += gs - gdd;
  return f0 + v;
}

// Both sides of one field's flux at x_{i+1/2}: returns f-hat = f-hat^+ +
// f-hat^-; gp (6: f^+ at i-1..i+1, H^+ at i-1..i+1) and gm (6: f^- at i..i+2,
// H^- at i..i+2) receive mu times the partial derivatives. The "-" side is
// the mirror image (reversed stencil, negated H).
__device__ __forceinline__ double flux_vjp(const double* fp_, const double* Hp_, const double* fm_,
                                         const double* Hm_, double mu, const Weights<double>& w,
                                         double* gp, double* gm, bool frozen = false) {
  const double fp = side_vjp(fp_[0], fp_[1], fp_[2], Hp_[0], Hp_[1], Hp_[2], mu, w, gp, frozen);
  double r[6] = {0, 0, 0, 0, 0, 0};
  const double fm =
      side_vjp(fm_[2], fm_[1], fm_[0], -Hm_[2], -Hm_[1], -Hm_[0], mu, w, r, frozen);
  gm[0] += r[2]; gm[1] += r[1]; gm[2] += r[0];
  gm[3] -= r[5]; gm[4] -= r[4]; gm[5] -= r[3];
  return fp + fm;
}

// One side of flux_vjp: sd = 0 the "+" side from (f0, f1, f2, H0, H1, H2) =
// f^+, H^+ at i-1..i+1; sd = 1 the "-" side from f^-, H^- at i..i+2 (its
// mirror image). Returns the side's value and adds mu times its partial
// derivatives to g (f then H, in stencil order).
__device__ __forceinline__ double side_half(int sd, double f0, double f1, double f2, double H0,
                                          double H1, double H2, double mu,
                                          const Weights<double>& w, double* g,
                                          bool frozen = false) {
  double r[6] = {0, 0, 0, 0, 0, 0};
  const double v = side_vjp(sd ? f2 : f0, f1, sd ? f0 : f2, sd ? -H2 : H0, sd ? -H1 : H1,
                            sd ? -H0 : H2, mu, w, r, frozen);
  if (sd) {
    g[0] += r[2]; g[1] += r[1]; g[2] += r[0];
    g[3] -= r[5]; g[4] -= r[4]; g[5] -= r[3];
  } else {
#pragma unroll
    for (int k = 0; k < 6; ++k) g[k] += r[k];
  }
  return v;
}

// Linear derivative flux D = dx (h-hat^+ + h-hat^-) (Sec. 2.1, p_0'):
// adds mu * dD/d input to gp, gm (same layout as flux_vjp).
__device__ __forceinline__ void dflux_vjp(double mu, double* gp, double* gm) {
  gp[0] += 0.25 * mu; gp[1] += -2.0 * mu; gp[2] += 1.75 * mu;
  const double x = 1.0 / 12.0 * mu;
  gp[3] += x; gp[4] -= 2.0 * x; gp[5] -= 5.0 * x;
  gm[0] += -1.75 * mu; gm[1] += 2.0 * mu; gm[2] += -0.25 * mu;
  gm[3] -= 5.0 * x; gm[4] -= 2.0 * x; gm[5] += x;
}

// HWENO limiter (Sec. 2.2) in scaled form, out = dx v-tilde from point values
// um, u0, up and Vm = dx v_{i-1}, Vp = dx v_{i+1}: returns out and adds
// mu * d out / d input to g[5] (order um, u0, up, Vm, Vp).
__device__ __forceinline__ double limiter_vjp(double um, double u0, double up, double Vm, double Vp,
                                            double mu, const Weights<double>& w, double* g,
                                            bool frozen = false) {
  using namespace adj;
  const double q1 = u0 - um, q2 = up - u0, lap = q2 - q1, du = q1 + q2;
  const double sV = Vm + Vp, dV = Vm - Vp, r = sV - du;
  const double z1 = r + L1 * du, z2 = dV + L2 * lap;
  const double c1 = LZ1 * z1, cu = LU * du, c2 = LZ2 * z2, cl = LL * lap;
  const double b0 = c1 * z1 + (cu * du + (c2 * z2 + (cl * lap + w.eps)));
  double gp0, gp1, gp2, gb0, gb1, gb2;
  const double v = weighted_vjp(b0, q1 * q1 + w.eps, q2 * q2 + w.eps, 0.75 * du - 0.25 * sV, q1, q2,
                                0.25 * r - 0.5 * lap, 0.25 * r + 0.5 * lap, -lap, w.d0, w.d1, w.d2,
                                mu, frozen, gp0, gp1, gp2, gb0, gb1, gb2);
  const double t0 = 2.0 * gb0;
  const double gz1 = t0 * c1, gdV = t0 * c2;
  const double gsV = gz1 - 0.25 * gp0;
  // the cotangents of q1 and q2 but for 3/4 gp0 of each, which is added last (one
  // rounding of the full value) and drops out of their difference
  const double gl = L2 * gdV + t0 * cl, gdu = (L1 - 1.0) * gz1 + t0 * cu;
  const double gq1 = 2.0 * (gb1 * q1) + (gp1 + (gdu - gl));
  const double gq2 = 2.0 * (gb2 * q2) + (gp2 + (gdu + gl));
  g[0] -= 0.75 * gp0 + gq1;
  g[1] += gq1 - gq2;
  g[2] += 0.75 * gp0 + gq2;
  g[3] += gsV + gdV;
  g[4] += gsV - gdV;
  return v;
}

}  // namespace hweno
