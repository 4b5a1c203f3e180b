"""The top of the persistent solve where gamma0 is small beside the contacts:
P^-1 then has eigenvalues of 1 / gamma0 (translations of a whole tree) beside
those of the contacts, and a rounded operator has to stay positive definite."""
from __future__ import annotations

import numpy as np
import pytest
import torch

import paper_2410_04512_gb300 as sgp
import workloads
from gpu_common import GpuSystem, dev_tensor

pytestmark = pytest.mark.gpu


def _sheet(gamma0):
    c = workloads.hex_sheet(nx=151, ny=133, seed=3007)
    return workloads.Cells("sheet", c.pos, c.radii, c.seed, c.gamma_lo, c.gamma_hi, gamma0)


def _balanced(n):
    """Internal forces: they sum to zero."""
    F = np.random.default_rng(17).standard_normal((n, 3))
    return dev_tensor(F - F.mean(0))


def _context(cap):
    cx = sgp.Context(0)
    cx.set_tuning(bin_cap=cap)
    return cx


@pytest.mark.parametrize("gamma0", [1e-4, 1e-8, 1e-10])
def test_mixed_solve_with_small_gamma0(cuda_device, gamma0):
    """What the level kernels solve, the persistent launch solves: the FP32
    preconditioner is an L D L^T of rounded factors in both.  (The counts
    differ by the rounding of the inner solves, a few percent.)"""
    c = _sheet(gamma0)
    F = _balanced(c.n)
    its = []
    for cap in (-1, 0):
        cx = _context(cap)
        s = GpuSystem(cx, c, precision=sgp.PREC_MIXED)
        v, info = cx.pcg_solve(s.M, s.Fac, F, tol=1e-9, precision=sgp.PREC_MIXED, maxit=60000)
        assert info.status == 0 and info.true_rel_residual <= 1e-9
        its.append(info.iterations)
    assert its[1] <= 1.25 * its[0], its


@pytest.mark.parametrize("gamma0", [1e-4, 1e-8, 1e-10])
def test_forest_solve_residual_with_small_gamma0(cuda_device, gamma0):
    """Substitution leaves a residual of a few eps |P| |x|, whatever 1 / gamma0
    is when the forces balance; the one-launch solve makes no more rounding
    errors on any path than the level kernels make (its products along the
    top are formed once), so within a factor of 4 the residuals are the same."""
    c = _sheet(gamma0)
    b = _balanced(c.n)
    res = []
    for cap in (-1, 0):
        cx = _context(cap)
        s = GpuSystem(cx, c)
        te = s.T.edge_ids().long()
        ij, B = s.ij[te].long(), s.M.edge_blocks()[0][te]
        x = cx.tree_apply(s.Fac, b)
        d = (B @ (x[ij[:, 0]] - x[ij[:, 1]])[:, :, None]).squeeze(2)
        y = (gamma0 * x).index_add_(0, ij[:, 0], d).index_add_(0, ij[:, 1], d, alpha=-1.0)
        res.append(float((y - b).norm() / b.norm()))
    assert res[1] <= 4 * res[0], res
