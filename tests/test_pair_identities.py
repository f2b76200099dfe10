"""The pair kernels take the smoothness indicators as sums of squares of
triangular factorisations and the nonlinear value as the linear one plus a
correction. This checks, without a GPU, that these forms equal the paper's
(Sec. 2.1, Eq. GHYZP, and Sec. 2.2) symbolically, with the rational constants
read from the kernel source.
"""
import os
import re

import pytest

sympy = pytest.importorskip("sympy")
from sympy import Rational as R, expand, nsimplify, simplify, symbols  # noqa: E402

SRC = os.path.join(os.path.dirname(__file__), os.pardir, "paper_2207_05258_gb300", "csrc",
                   "weno_df.cuh")


def constants(name):
    """The quotients of integers in the body of function `name`, in order."""
    with open(SRC) as f:
        text = f.read()
    body = text[text.index(" " + name + "("):]
    body = body[:body.index("\n}")]
    return [R(int(a), int(b)) for a, b in re.findall(r"c\((-?\d+)\.0 / (\d+)\.0\)", body)]


def test_reconstruction_indicators():
    fm, f0, fp, Hm, H0, Hp = symbols("fm f0 fp Hm H0 Hp")
    sH, dH, lp, dif = Hm + Hp, Hm - Hp, fm - 2 * f0 + fp, fm - fp
    a1 = R(19, 192) * sH + R(79, 48) * H0 + R(27, 64) * dif
    a2, a4 = R(3, 8) * dH + R(5, 4) * lp, -dH / 4 - lp / 2
    a3 = -(R(11, 24) * sH + R(17, 6) * H0) - R(15, 8) * dif
    a5 = sH / 4 + H0 + R(3, 4) * dif
    beta0 = ((a1 + a3 / 4 + a5 / 16) ** 2 + R(13, 3) * (a2 + R(63, 130) * a4) ** 2
             + R(781, 20) * (a3 + R(8825, 10934) * a5) ** 2 + R(1421461, 2275) * a4 ** 2
             + R(21520059541, 1377684) * a5 ** 2)
    y1, y2, s, d = fm - f0 + H0, f0 - fp + H0, Hm + Hp - 2 * H0, Hm - Hp
    g, lap = y1 + y2, y1 - y2
    k1, k2, c1, cg, c2, cl, ca, cb = constants("flux_indicators")
    b0 = (H0 ** 2 + c1 * (s + k1 * g) ** 2 + cg * g ** 2 + c2 * (d + k2 * lap) ** 2
          + cl * lap ** 2)
    assert expand(b0 - beta0) == 0
    assert expand(H0 ** 2 + ca * y1 ** 2 - H0 ** 2 - R(13, 3) * (H0 - f0 + fm) ** 2) == 0
    assert expand(H0 ** 2 + cb * y2 ** 2 - H0 ** 2 - R(13, 3) * (H0 + f0 - fp) ** 2) == 0
    # candidates relative to p_0 and to f_i
    p0 = R(11, 60) * (fm + fp) + R(19, 30) * f0 + (Hm - Hp) / 20 + H0 / 2
    p1, p2 = fm / 6 + R(5, 6) * f0 + R(2, 3) * H0, R(5, 6) * f0 + fp / 6 + H0 / 3
    m = d + 2 * lap
    assert expand(60 * (p1 - p0) - (5 * g - 3 * m)) == 0
    assert expand(60 * (p2 - p0) - (-5 * g - 3 * m)) == 0
    assert expand(6 * (p1 - f0) - (y1 + 3 * H0)) == 0 and expand(6 * (p2 - f0) - (3 * H0 - y2)) == 0
    assert expand(60 * (p0 - f0) - (11 * lap + 3 * d + 30 * H0)) == 0


def test_limiter_indicators():
    um, u0, up, Vm, Vp = symbols("um u0 up Vm Vp")
    a1 = -(Vm + Vp) / 4 + R(3, 4) * (up - um)
    a2, a3 = (Vm - Vp) / 4 + um - 2 * u0 + up, (Vm + Vp) / 4 + (um - up) / 4
    a4 = (Vp - Vm) / 4 - (um - 2 * u0 + up) / 2
    beta0 = ((a1 + a3 / 4) ** 2 + R(13, 3) * (a2 + R(63, 130) * a4) ** 2 + R(781, 20) * a3 ** 2
             + R(1421461, 2275) * a4 ** 2)
    q1, q2 = u0 - um, up - u0
    lap, du, dV = q2 - q1, q1 + q2, Vm - Vp
    r = Vm + Vp - du
    k1, k2, c1, cd, c2, cl = constants("limiter_indicators")
    b0 = c1 * (r + k1 * du) ** 2 + cd * du ** 2 + c2 * (dV + k2 * lap) ** 2 + cl * lap ** 2
    assert expand(b0 - beta0) == 0
    q0 = R(3, 4) * (up - um) - (Vm + Vp) / 4
    assert expand(4 * (q1 - q0) - (r - 2 * lap)) == 0
    assert expand(4 * (q2 - q0) - (r + 2 * lap)) == 0


def test_correction():
    b0, b1, b2, t, g1, g2, p0, p1, p2 = symbols("b0 b1 b2 t g1 g2 p0 p1 p2")
    g0 = 1 - g1 - g2
    w = [g * (1 + t / b) for g, b in ((g0, b0), (g1, b1), (g2, b2))]
    value = (w[0] * (p0 - g1 * p1 - g2 * p2) / g0 + w[1] * p1 + w[2] * p2) / sum(w)
    den = b1 * b2 * (b0 + g0 * t) + t * b0 * (g1 * b2 + g2 * b1)
    n1, n2 = g1 * b2 * (b0 - b1), g2 * b1 * (b0 - b2)
    assert simplify(value - p0 - t * (n1 * (p1 - p0) + n2 * (p2 - p0)) / den) == 0
    # the two candidates as p and q of correction(): p1 - p0 = p + q, p2 - p0 = q - p
    p, q = symbols("p q")
    assert expand(n1 * (p + q) + n2 * (q - p) - (p * (n1 - n2) + q * (n1 + n2))) == 0


def test_derivative_flux():
    F, U, h, v = (symbols("%s:4" % c) for c in "FUhv")
    al, dx = symbols("alpha dx")
    f = {s: [(F[i] + s * al * U[i]) / 2 for i in range(4)] for s in (1, -1)}
    H = {s: [dx * (h[i] + s * al * v[i]) / 2 for i in range(4)] for s in (1, -1)}

    def dp0(a, b):
        return (a[0] - 8 * a[1] + 7 * a[2]) / 4 + (b[0] - 2 * b[1] - 5 * b[2]) / 12

    both = dp0(f[1][:3], H[1][:3]) - dp0(f[-1][:0:-1], [-x for x in H[-1][:0:-1]])
    form = (nsimplify(1.875) * (F[2] - F[1]) - (F[3] - F[0]) / 8
            + al / 8 * ((U[3] - U[2]) - (U[1] - U[0]))
            + dx / 24 * (h[0] + h[3] - 7 * (h[1] + h[2]))
            + al * dx / 24 * (v[0] - v[3] + 3 * (v[1] - v[2])))
    assert expand(both - form) == 0


def test_derivative_flux():
    """One side's dx p_0' from its differences, and the sum over both sides
    with the "-" side's rows reversed and negated, against the form in F, U, h,
    N that the FP64 path evaluates."""
    dx, al = symbols("dx alpha")
    F, U, h, N = (symbols(f"{q}m {q}k {q}p {q}q") for q in "FUhN")
    t0, t1 = F[2] - F[1], F[3] - F[0]
    su = (U[3] - U[2]) - (U[1] - U[0])
    sh = (h[0] + h[3]) - 7 * (h[1] + h[2])
    sv = 3 * (N[1] - N[2]) + N[0] - N[3]
    ref = (R(15, 8) * t0 - t1 / 8 + al / 8 * su + dx / 24 * (sh + al * sv))

    def side(sg, linear=False):  # rows of the "+" side, of the "-" side negated and reversed
        order = [0, 1, 2] if sg > 0 else [3, 2, 1]
        f = [(F[i] + sg * al * U[i]) / 2 for i in order]
        H = [sg * dx * (h[i] + sg * al * N[i]) / 2 for i in order]
        y1, y2 = f[1] - f[0], f[2] - f[1]  # edge rows (reversal and negation cancel)
        y1, y2 = H[1] - y1, H[1] - y2
        s, d = H[0] + H[2] - 2 * H[1], H[0] - H[2]
        if linear:
            return 11 * y1 + 19 * y2 + 3 * d
        return H[1] + (y1 + d - 7 * y2) / 4 - s / 6

    assert expand(side(1) - side(-1) - ref) == 0

    # the linear part of c: in FP64, and from the sides' differences
    lin = (11 * ((F[3] - F[2]) - (F[1] - F[0]))
           + al * (dx * (27 * (N[1] + N[2]) + 3 * (N[0] + N[3]))
                   - 27 * (U[2] - U[1]) - 11 * (U[3] - U[0]))
           + dx * (33 * (h[1] - h[2]) + 3 * (h[0] - h[3]))) / 120
    assert expand((side(1, True) + side(-1, True)) / 60 - lin) == 0
    with open(SRC) as fh:
        assert constants("derivative_part") == [R(-2, 3)] and "madd(Num<X>::c" in fh.read()


def test_weights_over_common_denominator():
    """The reverse mode's form: v = sum of phi_l p_l is the paper's combination,
    and the cotangents of the b_l are its derivatives (b_0 above the others, so
    that tau = (b_0 - (b_1 + b_2) / 2)^2; exact at rational points)."""
    b0, b1, b2, p0, p1, p2 = symbols("b0 b1 b2 p0 p1 p2")
    g1, g2 = R(1, 7), R(2, 5)
    g0 = 1 - g1 - g2
    e1, e2 = b0 - b1, b0 - b2
    ht = (e1 + e2) / 2
    tau = ht ** 2
    o = [g * (1 + tau / b) for g, b in ((g0, b0), (g1, b1), (g2, b2))]
    paper = (o[0] * (p0 - g1 * p1 - g2 * p2) / g0 + o[1] * p1 + o[2] * p2) / sum(o)
    q1, q2 = g1 * b2, g2 * b1
    n1, n2, b12, bt = q1 * e1, q2 * e2, b1 * b2, b0 + tau
    m = 1 / (b12 * (b0 + g0 * tau) + tau * b0 * (q1 + q2))
    f0, f1, f2 = b12 * bt * m, tau * m * n1, tau * m * n2
    P1, P2, P = p1 - p0, p2 - p0, p1 - p2
    r0, r1, r2 = -(f1 * P1 + f2 * P2), f0 * P1 + f2 * P, f0 * P2 - f1 * P
    gt = ht * m * (r0 * b12 + r1 * n1 + r2 * n2)
    k = m * r0 * bt - m * tau * (g1 * r1 + g2 * r2)
    grads = {b0: m * r0 * b12 + m * tau * (r1 * q1 + r2 * q2) + 2 * gt,
             b1: b2 * k + g2 * m * tau * b0 * r2 - gt,
             b2: b1 * k + g1 * m * tau * b0 * r1 - gt}
    for vals in ((9, 2, 3, 1, 4, -2), (5, 4, 1, -3, R(1, 2), 7)):
        at = dict(zip((b0, b1, b2, p0, p1, p2), vals))
        assert (paper - (f0 * p0 + f1 * p1 + f2 * p2)).subs(at) == 0
        assert (f0 + f1 + f2).subs(at) == 1
        for b, g in grads.items():
            assert (paper.diff(b) - g).subs(at) == 0
