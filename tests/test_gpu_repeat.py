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
