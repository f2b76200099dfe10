"""The large tiles that big FP64 launches take (256 threads: 252 points of a
line in 1D and the x-sweep, 8 columns x 31 rows in the y-sweep) at the smallest
launches that take them, with ragged last tiles: 2D against the oracle with the
tolerances of the 2D parity tests, 1D the same bits as another tile shape
(which the 1D cases compare with the oracle).
"""
import pytest
import torch

from test_gpu_pairs import dev, euler, hw  # noqa: F401
from test_gpu_pairs_2d import check_rhs, make_w, state

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", ["smooth", "jump", "noise"])
@pytest.mark.parametrize("eq", ["euler", "burgers"])
def test_sweeps(hw, eq, kind):  # noqa: F811
    nx, ny = 996, 311  # x: 4 segments (the last of 240); y: 125 x 11 blocks (4 columns, 1 row)
    U, V, Wd = state(nx, ny, kind)
    if eq == "burgers":
        U, V, Wd = U[:1] - 0.7, V[:1], Wd[:1]
    check_rhs(hw, make_w(eq, nx, ny, U, V, Wd, x1=2.0, y1=2.0))


@pytest.mark.parametrize("jumps,noise", [(2, 0.0), (0, 0.3)])
def test_batch(hw, jumps, noise):  # noqa: F811
    w = euler([497] * 612, 61, jumps, noise)
    out = []
    for v in (0, 1):
        s = hw.Solver.from_workload(w, tile_variant=v)
        out.append(s.rhs(dev(w.U), dev(w.V)))
        s.sync_status()
    assert all(torch.equal(out[0][k], out[1][k]) for k in out[0])
