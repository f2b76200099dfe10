"""The rule that sends a tile's listed items to groups of lanes or to one thread
each (line_df.cuh)."""
import pytest

import _host_build as H


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    return H.load(tmp_path_factory.mktemp("host"))


def test_group_rule(lib):
    """Listed items go to groups of lanes while that is less work for the FP64
    pipe of a sub-partition than one item per thread: four warps of 32 items take
    one item's time, 16 groups of interfaces (Euler: 4 to a warp) three warps'."""
    assert all(lib.host_few(3, 0, n) for n in (0, 1, 16, 48))
    assert not any(lib.host_few(3, 0, n) for n in (49, 64, 100, 125, 128, 200, 253))
    assert all(lib.host_few(3, 1, n) for n in (0, 8, 64)) and not lib.host_few(3, 1, 125)
    assert lib.host_few(1, 0, 32) and not lib.host_few(1, 0, 128)
