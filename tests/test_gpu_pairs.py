"""The FP64 stage kernels evaluate interfaces and limiter points in pairs of
FP32 numbers where the nonlinear correction is small and in FP64 elsewhere
(by groups of lanes when a tile has few such items, by one thread each when
it has many). These cases drive every route, its edges and its range against
the oracle: noise (every item in FP64), a single jump in a smooth field (a few
items), data scaled towards and past both ends of the pairs' range, and the
options that change the route.

Tolerance: that of the 1D parity tests, 1e-13 of the split-flux scale over dx
(L^1), over dx^2 (L^2) and of the state over dx (v~): a few hundred units in
the last place of the terms that are differenced. A pair's own error, 2^-46 of
a correction that is at most 1/32 of the differences, is 4e-16 of them.
"""
import numpy as np
import pytest
import torch

from paper_2207_05258_gb300 import workloads as W
from test_gpu_parity_1d import SIZES, check_rhs, dev, hw  # noqa: F401

pytestmark = pytest.mark.gpu


def euler(sizes, seed, jumps, noise, scale=1.0, bc="outflow"):
    """Smooth waves with `jumps` density and pressure jumps and white noise of
    relative amplitude `noise`; rho, rho u and E scaled by `scale`."""
    g = np.random.default_rng(seed)
    Us, Vs = [], []
    for n in sizes:
        x = W.centers(0, 1, n)
        rho, drho = 1 + 0.2 * np.sin(2 * np.pi * x), 0.4 * np.pi * np.cos(2 * np.pi * x)
        p = 1 + 0.1 * np.cos(2 * np.pi * x)
        for x0 in g.uniform(0.1, 0.9, jumps):
            f = g.uniform(0.3, 3.0)
            rho, drho = np.where(x < x0, rho, f * rho), np.where(x < x0, drho, f * drho)
            p = np.where(x < x0, p, 0.7 * f * p)
        rho = rho * (1 + noise * g.uniform(-1, 1, n))
        u = 0.3 + noise * g.uniform(-1, 1, n)
        U = W.euler_conserved(rho, u, p, 1.4)
        V = np.stack([drho, 0.3 * drho, 0.05 * drho]) + noise * n * g.uniform(-1, 1, (3, n))
        Us.append(scale * U.ravel())
        Vs.append(scale * V.ravel())
    return W.Workload("pairs", "euler", 1, list(sizes), 1, 0.0, 1.0, 0.0, 1.0, 1.0,
                      (bc, bc, "periodic", "periodic"), np.concatenate(Us), np.concatenate(Vs))


def burgers(sizes, seed, jumps, noise, scale=1.0):
    g = np.random.default_rng(seed)
    Us, Vs = [], []
    for n in sizes:
        x = W.centers(0, 2, n)
        u = 0.5 + np.sin(np.pi * x) + noise * g.uniform(-1, 1, n)
        for x0 in g.uniform(0.2, 1.8, jumps):
            u = u + np.where(x < x0, 0.0, g.uniform(-1, 1))
        Us.append(scale * u)
        Vs.append(scale * (np.pi * np.cos(np.pi * x) + noise * n * g.uniform(-1, 1, n)))
    return W.Workload("pairs", "burgers", 1, list(sizes), 1, 0.0, 2.0, 0.0, 1.0, 1.0,
                      ("periodic",) * 4, np.concatenate(Us), np.concatenate(Vs))


@pytest.mark.parametrize("jumps,noise", [(0, 0.0), (1, 0.0), (6, 0.0), (0, 1e-3), (0, 0.3)])
def test_items_few_to_all(hw, jumps, noise):  # noqa: F811
    check_rhs(hw, euler(SIZES + [508, 997], 31 + jumps, jumps, noise))
    check_rhs(hw, burgers(SIZES + [508, 997], 41 + jumps, jumps, noise))


@pytest.mark.parametrize("variant", range(1, 5))
def test_tile_shapes(hw, variant):  # noqa: F811
    """Every tile shape gives the bits of the default one (which the other
    cases compare with the oracle)."""
    for jumps, noise in ((2, 0.0), (0, 0.3)):
        w = euler([59, 60, 61, 251, 252, 253, 504], 51, jumps, noise)
        out = []
        for v in (0, variant):
            s = hw.Solver.from_workload(w, tile_variant=v)
            out.append(s.rhs(dev(w.U), dev(w.V)))
            s.sync_status()
        assert all(torch.equal(out[0][k], out[1][k]) for k in out[0])


# the pairs take differences from 2^-126 to 2^40 and densities and wave speeds
# from 2^-30; beyond, FP64
@pytest.mark.parametrize("scale", [1e-40, 2e-10, 1e-9, 1e-3, 1e9, 1e11, 1e12, 1e13, 1e30])
def test_range(hw, scale):  # noqa: F811
    check_rhs(hw, euler([5, 100, 250], 61, 2, 0.0, scale))
    check_rhs(hw, euler([5, 100, 250], 62, 0, 0.2, scale))
    check_rhs(hw, burgers([5, 100, 250], 63, 2, 0.0, min(scale, 1e14)))


@pytest.mark.parametrize("opts", [dict(eig_avg=1), dict(limiter=0), dict(limiter=2),
                                  dict(eps=1e-20), dict(eps=1e6),
                                  dict(lin_w=(1 / 3, 1 / 3, 1 / 3), lim_d=(0.01, 0.495, 0.495)),
                                  dict(lin_w=(1 - 2e-6, 1e-6, 1e-6))])
def test_options(hw, opts):  # noqa: F811
    for jumps, noise in ((2, 0.0), (0, 0.2)):
        check_rhs(hw, euler([64, 129, 300], 71, jumps, noise, bc="reflective"), **opts)
        check_rhs(hw, burgers([64, 129, 300], 72, jumps, noise),
                  **{k: v for k, v in opts.items() if k != "eig_avg"})


@pytest.mark.parametrize("n", [31, 60, 61, 124, 200, 400, 420, 960, 961, 992])
def test_cluster_step_is_the_tiled_step(hw, n):  # noqa: F811
    """The wide form (cluster step of the scalar equations and of larger Euler
    instances; tiled stages that leave SMs idle) gives the bits of the tiled
    form (a batch too large for the wide form)."""
    for w1, big in ((burgers([n], 81, 1, 0.0), burgers([n] + [125] * 200, 81, 1, 0.0)),
                    (euler([n], 82, 2, 0.01), euler([n] + [125] * 200, 82, 2, 0.01))):
        out = []
        for w, opts in ((w1, {}), (w1, dict(fused_small=2)), (big, {})):
            if w.equation == "euler" and n <= 448 and opts:
                continue  # the latency form, compared with the oracle elsewhere
            s = hw.Solver.from_workload(w, cfl=0.4, **opts)
            U, V = dev(w.U), dev(w.V)
            t = torch.zeros(w.batch, dtype=torch.float64, device="cuda")
            for _ in range(3):
                s.step(U, V, None, t, 1e30)
            s.sync_status()
            m = w.m * n
            out.append((U[:m].clone(), V[:m].clone(), t[:1].clone()))
        for o in out[1:]:
            assert all(torch.equal(a, b) for a, b in zip(out[0], o))
