"""Repeated solves give the same bits, on every path that sums across rows:
the multi-launch FP64 step from 100,000 rows on (rows dealt to lanes by
length), and the persistent launch with the factor rebuilt (parts dealt from
lists that atomics fill)."""
from __future__ import annotations

import numpy as np
import pytest
import torch

import paper_2410_04512_gb300 as sgp
import workloads
from gpu_common import GpuSystem, dev_tensor
from test_gpu_batched import GpuBatch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precond", [sgp.PRECOND_TREE, sgp.PRECOND_NONE])
def test_multi_launch_fp64_steps_repeat(cuda_device, precond):
    """p^T q, and with it every iterate, does not depend on timing."""
    c = workloads.hex_sheet(nx=331, ny=311, seed=3)   # 102,941 cells
    F = dev_tensor(c.forces())
    cx = sgp.Context(0)
    cx.set_tuning(bin_cap=-1)
    s = GpuSystem(cx, c, tree=precond == sgp.PRECOND_TREE)
    first = None
    for _ in range(6):
        v, info = cx.pcg_solve(s.M, s.Fac, F, tol=1e-300, maxit=30, precond=precond, raise_on_error=False)
        assert info.iterations == 30
        if first is None:
            first = v.clone()
        assert torch.equal(v, first)


@pytest.mark.parametrize("precision", [sgp.PREC_F64, sgp.PREC_MIXED])
@pytest.mark.parametrize("what", ["tree", "jacobi", "none", "batch", "network", "apply"])
def test_persistent_launches_repeat(cuda_device, what, precision):
    """The same bits again, and after the factor is built again."""
    cx = sgp.Context(0)
    if what == "batch":
        b = GpuBatch(cx, [3000, 2600, 0, 4000], precision=precision)
        F = dev_tensor(b.F)
        M, T, Fac = b.M, b.T, b.Fh

        def run():
            return cx.pcg_solve_batched(M, Fac, b.off, F, tol=1e-10, precision=precision)[0]
    else:
        c = workloads.ball(n=61003, seed=2110, gamma0=1e-3)
        F = dev_tensor(c.forces())
        s = GpuSystem(cx, c, precision=precision)
        M, T, Fac = s.M, s.T, s.Fac
        pre = {"tree": sgp.PRECOND_TREE, "jacobi": sgp.PRECOND_BLOCK_JACOBI, "none": sgp.PRECOND_NONE}.get(what)
        net = cx.mpnn_create((0.1 * np.random.default_rng(1).standard_normal(sgp.MPNN_PARAMS)).astype(np.float32))

        def run():
            if what == "apply":
                return cx.tree_apply(Fac, F)
            if what == "network":
                return cx.mpnn_forward(net, M, Fac, F)
            return cx.pcg_solve(M, Fac, F, tol=1e-10, precond=pre, precision=precision)[0]

    first = run().clone()
    for k in range(4):
        if k == 2:
            cx.tree_factor(M, T, Fac)
        assert torch.equal(run(), first)


@pytest.mark.parametrize("geometry", ["ball", "sheet"])
def test_multi_launch_fp64_steps_repeat_and_agree(cuda_device, geometry):
    """Rows of many lengths (a ball: dealt to lanes by length) and rows about
    equally long (a sheet: in their own order): the same bits in every run, and
    20 unpreconditioned steps equal to the one-launch solve's but for the order
    of sums (1e-10 of the iterate)."""
    c = workloads.ball(n=120011, seed=2120, gamma0=1e-3) if geometry == "ball" else workloads.hex_sheet(nx=331, ny=311, seed=3)
    F = dev_tensor(c.forces())
    out = []
    for cap in (0, -1):
        cx = sgp.Context(0)
        cx.set_tuning(bin_cap=cap)
        s = GpuSystem(cx, c, tree=False)
        kw = dict(tol=1e-300, maxit=20, precond=sgp.PRECOND_NONE, raise_on_error=False)
        out.append(cx.pcg_solve(s.M, None, F, **kw)[0].clone())
        for _ in range(4):
            assert torch.equal(cx.pcg_solve(s.M, None, F, **kw)[0], out[-1])
    assert float((out[0] - out[1]).norm() / out[1].norm()) <= 1e-10
