"""Rounding of the FP64 product against the same sum in extended precision."""
from __future__ import annotations

import numpy as np
import pytest

import paper_2410_04512_gb300 as sgp
import workloads
from gpu_common import GpuSystem, dev_tensor

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [60000, 120000])   # blocks of 128 and of 1024 rows
def test_rounding_of_the_product(cuda_device, n):
    """No further off than with each contact's products summed first and then
    added to the row in order (fused multiply-adds, as the compiler contracts
    them: emulated here by rounding once from extended precision)."""
    if np.finfo(np.longdouble).nmant < 63:
        pytest.skip("no extended precision here")
    c = workloads.ball(n=n, seed=2119, gamma0=1e-3)
    s = GpuSystem(sgp.Context(0), c)
    v = np.random.default_rng(6).standard_normal((n, 3))
    y = s.ctx.spmv(s.M, dev_tensor(v)).cpu().numpy()
    ij = s.ij.cpu().numpy()
    B = s.M.edge_blocks()[0].cpu().numpy().reshape(-1, 3, 3)
    L = np.longdouble
    rows = np.concatenate([ij[:, 0], ij[:, 1]])
    order = np.argsort(rows, kind="stable")
    rows = rows[order]
    d = v[ij[:, 0]] - v[ij[:, 1]]
    d = np.concatenate([d, -d])[order]
    dl = v[ij[:, 0]].astype(L) - v[ij[:, 1]].astype(L)
    dl = np.concatenate([dl, -dl])[order]
    B = np.concatenate([B, B])[order]
    exact = np.array(L(c.gamma0) * v.astype(L))
    t = B[:, :, 0] * d[:, 0:1]
    e = B[:, :, 0].astype(L) * dl[:, 0:1]
    for k in (1, 2):
        t = (B[:, :, k].astype(L) * d[:, k:k + 1] + t).astype(np.float64)
        e = e + B[:, :, k].astype(L) * dl[:, k:k + 1]
    np.add.at(exact, rows, e)
    plain = c.gamma0 * v
    np.add.at(plain, rows, t)
    size = np.sqrt((exact * exact).sum())
    off = [float(np.sqrt(((x - exact) ** 2).sum()) / size) for x in (y, plain)]
    assert off[0] <= off[1], off
