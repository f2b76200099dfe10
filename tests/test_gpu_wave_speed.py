"""The wave speeds of the stage outputs (evaluated in FP64 only where an FP32
value comes near the tile's largest) in steps of data at the ends of the FP32
range, against the oracle: supersonic cross-flow beside still gas, whose squared
momenta fall under the FP32 range while the state does not. Steps of other
parts of the state differ by the rounding of two orders of the same operations
(a few 1e-16 times the ten-odd operations of a stage and three stages); a wave
speed that is off shows as a difference of order one.
"""
import numpy as np
import pytest
import torch

import oracle as O
from _util import oracle_problem
from paper_2207_05258_gb300 import workloads as W
from test_gpu_parity_2d import dev, hw, make_w  # noqa: F401

pytestmark = pytest.mark.gpu
TOL = 1e-11


@pytest.mark.parametrize("scale", [1e-30, 1e-25, 1e-23, 1.0, 1e25])
@pytest.mark.parametrize("turn", [False, True])
def test_step_2d(hw, scale, turn):  # noqa: F811
    nx, ny = 130, 37
    x = W.centers(0, 1, nx)[None, :] + 0 * W.centers(0, 1, ny)[:, None]
    left = x < 0.5
    rho, one = np.ones_like(x), np.ones_like(x)
    u, v, p = one, np.where(left, 3.0, 0.0), np.where(left, 0.3, 1.0)
    if turn:
        u, v = v, u
    U = scale * W.euler_conserved(rho, u, p, 1.4, v=v)
    w = make_w("euler", nx, ny, U, 0 * U, 0 * U, bc=("outflow",) * 4)
    s = hw.Solver.from_workload(w)
    g = [dev(a) for a in (w.U, w.V, w.W)]
    t = torch.zeros(1, dtype=torch.float64, device="cuda")
    # (the gas streams colliding: in small units eps makes the weights linear,
    # with which the second step leaves the physical states, the oracle's too)
    steps = 1 if turn else 2
    for _ in range(steps):
        s.step(*g, t, 1e30)
    s.sync_status()
    ref = O.run(oracle_problem(w), w.U, w.V, w.W, 0.0, 1e30, max_steps=steps)
    assert abs(t.item() - ref[3]) <= 1e-13 * ref[3]
    for a, b, size in zip(g, ref[:3], (1, nx, nx)):  # derivatives: of the size of U / h
        e = np.abs(a.cpu().numpy() - np.asarray(b).ravel()).max() / (size * np.abs(U).max())
        assert e <= TOL, e
