"""The reverse mode of one side's flux and of the limiter (hweno_adjoint.cuh)
against forward-mode differentiation of the paper's formulas (Sec. 2.1-2.2) in
long double, over the range of the data.

Tolerance: a gradient is about 100 operations, each rounding sums that exceed
their result by the largest coefficient of the indicators over the others
(about 1e3 / 4): 100 * 250 * 1.1e-16 = 3e-12 of the stencil's largest partial
derivative.
"""
import numpy as np
import pytest

import _host_build as H

TOL = 3e-12
L = np.longdouble


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    return H.load(tmp_path_factory.mktemp("host"))


class Dual:
    """Arrays of values with k tangents."""

    def __init__(self, v, d):
        self.v, self.d = v, d

    def __add__(self, o):
        return Dual(self.v + o.v, self.d + o.d) if isinstance(o, Dual) else Dual(self.v + o, self.d)

    def __mul__(self, o):
        if isinstance(o, Dual):
            return Dual(self.v * o.v, self.d * o.v + self.v * o.d)
        return Dual(self.v * o, self.d * o)

    def __neg__(self):
        return self * L(-1)

    def __sub__(self, o):
        return self + (-o)

    def inv(self):
        return Dual(1 / self.v, -self.d / self.v / self.v)

    def abs(self):
        return Dual(np.abs(self.v), self.d * np.sign(self.v))

    __radd__, __rmul__ = __add__, __mul__


def q(a, b):
    return L(a) / L(b)


def weights(b, p, g, eps):
    """(w_0 (p_0 - g_1 p_1 - g_2 p_2) / g_0 + w_1 p_1 + w_2 p_2) / sum w."""
    t = ((b[0] - b[1]).abs() + (b[0] - b[2]).abs()) * q(1, 2)
    tau = t * t
    w = [(tau * (x + eps).inv() + L(1)) * gg for x, gg in zip(b, g)]
    s = (w[0] + w[1] + w[2]).inv()
    r = (p[0] - p[1] * g[1] - p[2] * g[2]) * (1 / g[0])
    return (w[0] * r + w[1] * p[1] + w[2] * p[2]) * s


def side(x, g, eps):
    fm, f0, fp, Hm, H0, Hp = x
    sH, dH, lp, dif = Hm + Hp, Hm - Hp, fm - f0 * L(2) + fp, fm - fp
    # beta_0 in the a_l of the quintic; e_1 = a_1 + a_3 / 4 + a_5 / 16 = H_i
    a2, a4 = dH * q(3, 8) + lp * q(5, 4), -dH * q(1, 4) - lp * q(1, 2)
    a3 = -(sH * q(11, 24) + H0 * q(17, 6)) - dif * q(15, 8)
    a5 = sH * q(1, 4) + H0 + dif * q(3, 4)
    e2, e3 = a2 + a4 * q(63, 130), a3 + a5 * q(8825, 10934)
    b0 = (H0 * H0 + e2 * e2 * q(13, 3) + e3 * e3 * q(781, 20) + a4 * a4 * q(1421461, 2275)
          + a5 * a5 * q(21520059541, 1377684))
    s1, s2 = H0 - f0 + fm, H0 + f0 - fp
    b = [b0, H0 * H0 + s1 * s1 * q(13, 3), H0 * H0 + s2 * s2 * q(13, 3)]
    p = [(fm + fp) * q(11, 60) + f0 * q(19, 30) + dH * q(1, 20) + H0 * q(1, 2),
         fm * q(1, 6) + f0 * q(5, 6) + H0 * q(2, 3), f0 * q(5, 6) + fp * q(1, 6) + H0 * q(1, 3)]
    return weights(b, p, g, eps)


def limiter(x, g, eps):
    um, u0, up, Vm, Vp = x[:5]
    sV, dV, lp, du = Vm + Vp, Vm - Vp, um - u0 * L(2) + up, up - um
    q0 = du * q(3, 4) - sV * q(1, 4)
    a2, a3 = dV * q(1, 4) + lp, sV * q(1, 4) - du * q(1, 4)
    a4 = -dV * q(1, 4) - lp * q(1, 2)
    e1, e2 = q0 + a3 * q(1, 4), a2 + a4 * q(63, 130)
    b0 = e1 * e1 + e2 * e2 * q(13, 3) + a3 * a3 * q(781, 20) + a4 * a4 * q(1421461, 2275)
    q1, q2 = u0 - um, up - u0
    return weights([b0, q1 * q1, q2 * q2], [q0, q1, q2], g, eps)


def stencils(kind, scale, n=400):
    g = np.random.default_rng(3)
    if kind == "noise":
        x = g.uniform(-1, 1, (n, 6))
    else:  # a wave, its derivatives to match; a jump on one side. (Not a parabola:
        # its three indicators are equal, where tau's |.| have their kinks.)
        a, b, c = (g.uniform(-1, 1, (n, 1)) for _ in range(3))
        z, h = np.array([-1.0, 0.0, 1.0]), 0.5
        x = np.hstack([a + b * np.sin(h * z + 3 * c), h * b * np.cos(h * z + 3 * c)])
        if kind == "jump":
            x[:, 2] += g.uniform(0.5, 1, n)
    return np.ascontiguousarray(x * scale)


@pytest.mark.parametrize("kind", ["smooth", "jump", "noise"])
@pytest.mark.parametrize("scale", [1e-20, 1e-3, 1.0, 1e3, 1e20, 1e35, 1e37, 1e38, 1e48, 1e80, 1e130])
@pytest.mark.parametrize("which", [side, limiter])
def test_gradient(lib, which, scale, kind):
    x = stencils(kind, scale)
    w, eps = np.array([0.98, 0.01, 0.01]), 1e-6
    v, g = np.zeros(len(x)), np.zeros_like(x)
    lib.host_vjp(int(which is limiter), len(x), H.ptr(x), H.ptr(w), H.ctypes.c_double(eps), H.ptr(v),
                 H.ptr(g))
    d = np.eye(6, dtype=L)
    ref = which([Dual(x[:, k].astype(L), np.repeat(d[:, k:k + 1], len(x), 1)) for k in range(6)],
                w.astype(L), L(eps))
    assert np.isfinite(g).all() and np.isfinite(v).all()
    err = np.abs(g.T - ref.d).max(axis=0) / np.abs(ref.d).max(axis=0)
    assert err.max() <= TOL, err.max()
    assert (np.abs(v - ref.v) / np.abs(x).max(axis=1)).max() <= TOL


def test_limiter_gradient_of_smooth_data(lib):
    """Nearly the linear weights' gradient, (-3/4, 0, 3/4, -1/4, -1/4): each entry
    is rounded at most four times at its full size (phi_0, the product, the sum;
    root mean square 3.2e-17 each in [1/2, 1), half that in [1/4, 1/2)), the rest
    of it is small."""
    g = np.random.default_rng(4)
    a, b, c = (g.uniform(-1, 1, (20000, 1)) for _ in range(3))
    z = np.array([-0.05, 0.0, 0.05])
    x = np.ascontiguousarray(np.hstack([a + b * np.sin(z + 3 * c),
                                        0.05 * b * np.cos(z[[0, 2, 1]] + 3 * c)]))
    w, v, gr = np.array([0.98, 0.01, 0.01]), np.zeros(len(x)), np.zeros_like(x)
    lib.host_vjp(1, len(x), H.ptr(x), H.ptr(w), H.ctypes.c_double(1e-6), H.ptr(v), H.ptr(gr))
    d = np.eye(6, dtype=L)
    ref = limiter([Dual(x[:, k].astype(L), np.repeat(d[:, k:k + 1], len(x), 1)) for k in range(6)],
                  w.astype(L), L(1e-6))
    rms = np.sqrt(((gr.T - ref.d) ** 2).mean(axis=1))
    assert (rms[[0, 2]] <= 2 * 3.2e-17).all() and (rms[[3, 4]] <= 2 * 1.6e-17).all(), rms
    assert rms[1] <= 1e-18
