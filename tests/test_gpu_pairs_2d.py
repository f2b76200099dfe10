"""The FP64 2D sweeps (pairs of FP32 numbers for small corrections, FP64 for
the listed items) against the oracle at the edges of their tiles (x: 124
points of a row, y: 4 columns x 31 rows), with no, few and only listed items,
and at both ends of the pairs' range. Tolerances: those of the 2D parity tests
(1e-13 of the split-flux scale over the mesh widths).
"""
import numpy as np
import pytest

from paper_2207_05258_gb300 import workloads as W
from test_gpu_parity_2d import check_rhs, hw, make_w, rand_euler2d  # noqa: F401

pytestmark = pytest.mark.gpu
SIZES = [(4, 4), (5, 31), (3 + 124, 32), (124, 33), (125, 30), (249, 62), (9, 63)]


def state(nx, ny, kind):
    if kind == "noise":
        return rand_euler2d(nx, ny, nx + ny)
    w = W.euler2d_smooth(nx, ny)
    U, V, Wd = (a.reshape(4, ny, nx).copy() for a in (w.U, w.V, w.W))
    if kind == "jump":  # a jump across one column and one row
        f = np.ones((ny, nx))
        f[:, nx // 2:] *= 2.5
        f[ny // 2:] *= 0.4
        U, V, Wd = U * f, V * f, Wd * f
    return U, V, Wd


@pytest.mark.parametrize("kind", ["smooth", "jump", "noise"])
@pytest.mark.parametrize("nx,ny", SIZES)
def test_tile_edges(hw, nx, ny, kind):  # noqa: F811
    U, V, Wd = state(nx, ny, kind)
    check_rhs(hw, make_w("euler", nx, ny, U, V, Wd, x1=2.0, y1=2.0))
    check_rhs(hw, make_w("burgers", nx, ny, U[:1] - 0.7, V[:1], Wd[:1], x1=2.0, y1=2.0))


@pytest.mark.parametrize("scale", [1e-40, 1e-9, 1e11, 1e13, 1e30])
def test_range(hw, scale):  # noqa: F811
    for kind in ("jump", "noise"):
        U, V, Wd = (scale * a for a in state(66, 37, kind))
        check_rhs(hw, make_w("euler", 66, 37, U, V, Wd, bc=("outflow", "outflow", "reflective",
                                                            "reflective")))
