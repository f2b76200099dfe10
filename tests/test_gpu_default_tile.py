"""The tile shape that a context of a large FP64 Euler batch starts with: shown by
the options, kept when others are changed, replaced by the one asked for, and
with the results and sums of the 124-point shape."""
import pytest
import torch

from test_gpu_pairs import dev, euler, hw  # noqa: F401

pytestmark = pytest.mark.gpu


def test_default_tile(hw):  # noqa: F811
    w = euler([497] * 612, 61, 2, 0.0)  # the smallest such batch: 1 224 tiles of 252 points
    s = hw.Solver.from_workload(w)
    assert s.options().tile_variant == 2
    s.set_options(limiter=2)
    assert s.options().tile_variant == 2
    s.set_options(limiter=1)
    U, V = dev(w.U), dev(w.V)
    a, sums = s.rhs(U, V), s.totals(U)
    s.set_options(tile_variant=0)
    assert s.options().tile_variant == 0
    assert torch.equal(sums, s.totals(U))
    b = s.rhs(U, V)
    s.set_options(tile_variant=1)
    s.set_options(tile_variant=0)
    assert s.options().tile_variant == 0
    c = s.rhs(U, V)
    s.sync_status()
    assert all(torch.equal(a[k], b[k]) and torch.equal(a[k], c[k]) for k in a)
    for eq, precision, n in (("euler", "fp64", 607), ("euler", "fp32", 612), ("burgers", "fp64", 612)):
        assert hw.Solver(eq, 1, [497] * n, precision=precision).options().tile_variant == 0
