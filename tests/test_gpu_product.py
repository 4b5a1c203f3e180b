"""The FP64 product and the forest solve alone where their kernels change
shape: block edges, rows longer than the length buckets, the largest block."""
from __future__ import annotations

import numpy as np
import pytest
import torch

import oracle
import paper_2410_04512_gb300 as sgp
import workloads
from gpu_common import GpuSystem, dev_tensor, oracle_system, rel_err, small_cube
from test_gpu_grid import _cells

pytestmark = pytest.mark.gpu


def _shape(name):
    if name.startswith("cube"):
        return small_cube(int(name[4:]), seed=7)
    if name == "sheet100k":
        return workloads.hex_sheet(nx=331, ny=311, seed=3)
    return _cells(name)


@pytest.mark.parametrize("name", ["one", "cube127", "cube128", "cube129", "hub", "forest", "sheet100k"])
def test_product(cuda_device, name):
    """A row is at most a few thousand terms summed in FP64; each is accurate
    to a few 2^-53 of its own size, and the rows do not cancel as a whole
    (random v): 1e-12 of the norm is far above what rounding gives."""
    c = _shape(name)
    s = GpuSystem(sgp.Context(0), c)
    o = oracle_system(c)
    v = np.random.default_rng(3).standard_normal((c.n, 3))
    y = s.ctx.spmv(s.M, dev_tensor(v)).cpu().numpy()
    assert rel_err(y, oracle.matvec(c.n, o.ij, o.blocks, c.gamma0, v)) <= 1e-12


@pytest.mark.parametrize("name", ["hub", "chain", "forest", "sheet", "cube129", "ball"])
def test_forest_solve_alone(cuda_device, name):
    """One launch against the level kernels on the same factor values.  Both
    are backward stable (error about 1e-16 times the condition number, at most
    (gamma0 + lambda_max) / gamma0 < 1e6): 1e-10.  In place as well."""
    c = _cells(name)
    b = dev_tensor(np.random.default_rng(4).standard_normal((c.n, 3)))
    out = []
    for cap in (0, -1):
        cx = sgp.Context(0)
        cx.set_tuning(bin_cap=cap)
        s = GpuSystem(cx, c)
        out.append(cx.tree_apply(s.Fac, b).clone())
        w = b.clone()
        cx.tree_apply(s.Fac, w, w)
        assert torch.equal(w, out[-1])
    assert rel_err(out[0].cpu().numpy(), out[1].cpu().numpy()) <= 1e-10


def test_product_inside_multi_launch_steps(cuda_device):
    """From 100,000 rows on the multi-launch FP64 step takes the sorted product
    with p^T q: 20 unpreconditioned steps against the one-launch solve, equal
    but for the order of sums (1e-10 of the iterate)."""
    c = _shape("sheet100k")
    F = dev_tensor(c.forces())
    out = []
    for cap in (0, -1):
        cx = sgp.Context(0)
        cx.set_tuning(bin_cap=cap)
        s = GpuSystem(cx, c, tree=False)
        v, info = cx.pcg_solve(s.M, None, F, tol=1e-300, maxit=20, precond=sgp.PRECOND_NONE, raise_on_error=False)
        assert info.iterations == 20
        out.append(v.cpu().numpy())
    assert rel_err(out[0], out[1]) <= 1e-10
