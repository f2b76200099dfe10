"""The adjoint of a step of large data (split-flux jumps of 1e36 to 1e46) against
the oracle's forward-mode derivative, as test_gpu_adjoint.py does at unit scale
and to its tolerance."""
import numpy as np
import pytest
import torch

import oracle as O
from _util import oracle_problem
from test_gpu_adjoint import hw, rough_batch  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scale", [1e18, 3e18, 1e19, 1e21, 1e23])
def test_dot_product(hw, scale):  # noqa: F811
    w = rough_batch([31, 125], "periodic", 7)
    w.U[:] *= scale
    w.V[:] *= scale
    s = hw.Solver.from_workload(w)
    U, V = torch.from_numpy(w.U.copy()).cuda(), torch.from_numpy(w.V.copy()).cuda()
    t = torch.zeros(w.batch, dtype=torch.float64, device="cuda")
    dt = torch.empty_like(t)
    s.step(U.clone(), V.clone(), None, t, 1.0, dt)
    rng = np.random.default_rng(11)
    lamU, lamV = rng.standard_normal(w.U.size), rng.standard_normal(w.V.size)
    lU, lV = torch.from_numpy(lamU).cuda(), torch.from_numpy(lamV).cuda()
    s.adjoint_step(U, V, None, dt, lU, lV)
    s.sync_status()
    gU, gV = lU.cpu().numpy(), lV.cpu().numpy()
    off = 0
    for k, n in enumerate(w.nx):
        Uk, Vk = w.instance(k)
        dU, dV = rng.standard_normal(Uk.shape), rng.standard_normal(Vk.shape)
        out = O.run_tangent(oracle_problem(w, nx=n), Uk, Vk, None, dU, dV, None, 0.0, 1.0,
                            max_steps=1)
        part = slice(off, off + n)
        lhs = float(np.dot(gU[part], dU.ravel()) + np.dot(gV[part], dV.ravel()))
        rhs = float(np.dot(lamU[part], out[3].ravel()) + np.dot(lamV[part], out[4].ravel()))
        size = np.sqrt(np.sum(lamU[part] ** 2 + lamV[part] ** 2)
                       * np.sum(out[3] ** 2 + out[4] ** 2)) + abs(rhs)
        assert abs(lhs - rhs) <= 1e-12 * size, (scale, n, lhs, rhs)
        off += n
