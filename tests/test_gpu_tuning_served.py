"""The autotuner where one launch serves the whole solve: knobs that the launch
does not read are not chosen by chance between equal times."""
from __future__ import annotations

import pytest

import paper_2410_04512_gb300 as sgp
import workloads
from gpu_common import GpuSystem, dev_tensor
from test_gpu_batched import GpuBatch

pytestmark = pytest.mark.gpu

DEAD = ("spmv_lpr", "spmv_ilp", "tail_cap", "batch_chunk")


def test_batch_of_more_instances_than_blocks(cuda_device):
    """No persistent launch and no layout: every knob is timed."""
    cx = sgp.Context(0)
    b = GpuBatch(cx, [5] * 170, precision=sgp.PREC_MIXED)
    t = cx.autotune(b.M, b.T, b.Fh, dev_tensor(b.F), offsets=b.off, precision=sgp.PREC_MIXED, iterations=3)
    assert t["batch_chunk"] in (512, 1024, 2048, 4096, 8192) and cx.get_tuning()["batch_chunk"] == t["batch_chunk"]


@pytest.mark.parametrize("start", [{}, {"spmv_lpr": 4, "spmv_ilp": 2, "tail_cap": 512, "batch_chunk": 1024}])
@pytest.mark.parametrize("what", ["tree", "jacobi", "batch"])
def test_unread_knobs_stay(cuda_device, what, start):
    cx = sgp.Context(0)
    cx.set_tuning(**start)
    before = cx.get_tuning()
    if what == "batch":
        b = GpuBatch(cx, [3000, 2600, 4000], precision=sgp.PREC_MIXED)
        t = cx.autotune(b.M, b.T, b.Fh, dev_tensor(b.F), offsets=b.off, precision=sgp.PREC_MIXED, iterations=20)
    else:
        c = workloads.ball(n=30000, seed=2003, gamma0=1e-3)
        s = GpuSystem(cx, c, precision=sgp.PREC_MIXED, tree=what == "tree")
        pre = sgp.PRECOND_TREE if what == "tree" else sgp.PRECOND_BLOCK_JACOBI
        t = cx.autotune(s.M, s.T, s.Fac, dev_tensor(c.forces()), precond=pre, precision=sgp.PREC_MIXED, iterations=20)
    after = cx.get_tuning()
    assert t["bin_cap"] == 0 and t["ms_per_iteration"] > 0   # the persistent launch is the fastest by far here
    for k in DEAD:
        assert after[k] == before[k], k
    # what `out` says is in effect
    assert t["spmv_lpr"] == (before["spmv_lpr"] or 2) and t["spmv_ilp"] == (before["spmv_ilp"] or 1)
