"""The ways a tile's listed items are evaluated (groups of lanes, one thread per
item from rows of doubles; tiles of 64, 128 and 256 threads, the wide form) give
the same bits for any number of listed items, and those of the oracle to the 1D
parity tests' tolerance."""
import numpy as np
import pytest
import torch

from test_gpu_pairs import burgers, check_rhs, dev, euler, hw  # noqa: F401

pytestmark = pytest.mark.gpu
# 201 and more tiles of every shape (more than the wide form takes)
SIZES = [59, 60, 61, 251, 252, 253, 504] + [125] * 200


def outputs(hw, w, **opts):  # noqa: F811
    s = hw.Solver.from_workload(w, cfl=0.3, **opts)
    U, V = dev(w.U), dev(w.V)
    r = s.rhs(U, V)
    t = torch.zeros(w.batch, dtype=torch.float64, device="cuda")
    for _ in range(3):
        s.step(U, V, None, t, 1e30)
    s.sync_status()
    return [r["L1"], r["L2"], r["Vt"], U, V, t]


@pytest.mark.parametrize("variant", range(1, 5))
@pytest.mark.parametrize("make", [euler, burgers])
def test_tile_shapes(hw, make, variant):  # noqa: F811
    for jumps, noise in ((2, 0.0), (0, 0.05)):
        w = make(SIZES, 51, jumps, noise)
        for a, b in zip(outputs(hw, w), outputs(hw, w, tile_variant=variant)):
            assert torch.equal(a, b)


def part_noise(make, sizes, seed):
    """Instance k: the middle of a smooth field replaced by noise over k % 130
    points, so that every number of listed items occurs."""
    w, n = make(sizes, seed, 0, 0.0), make(sizes, seed, 0, 0.2)
    off = 0
    for k, size in enumerate(sizes):
        m = w.U.size // sum(sizes)
        for c in range(m):
            lo = off + c * size + max(0, (size - k % 130) // 2)
            hi = min(lo + k % 130, off + (c + 1) * size)
            w.U[lo:hi], w.V[lo:hi] = n.U[lo:hi], n.V[lo:hi]
        off += m * size
    return w


@pytest.mark.parametrize("make", [euler, burgers])
def test_any_number_of_listed_items(hw, make):  # noqa: F811
    w = part_noise(make, [124] * 130, 52)  # 130 tiles: the wide form
    check_rhs(hw, w)
    big = make([124] * 260, 52, 0, 0.0)  # the same instances in the tiled form
    big.U[:w.U.size], big.V[:w.V.size] = w.U, w.V
    s = [hw.Solver.from_workload(x) for x in (w, big)]
    r = [q.rhs(dev(x.U), dev(x.V)) for q, x in zip(s, (w, big))]
    for k in r[0]:
        assert torch.equal(r[0][k], r[1][k][:w.U.size])
