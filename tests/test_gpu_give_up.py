"""Bounded waits that give up: where one thread block of a persistent launch
numbers its packets wrongly, the waits for it run out, and each call says
TIMEOUT (not a breakdown, not a result)."""
from __future__ import annotations

import numpy as np
import pytest
import torch

import paper_2410_04512_gb300 as sgp
import workloads
from gpu_common import GpuSystem, dev_tensor
from test_gpu_batched import GpuBatch

pytestmark = pytest.mark.gpu


@pytest.fixture()
def skewed(cuda_device, monkeypatch):
    """A context whose waits run out (soon: its launches start with the word
    set that ends waits after some polls)."""
    monkeypatch.setenv("SGP_SKEW_PACKETS", "1")
    cx = sgp.Context(0)
    monkeypatch.delenv("SGP_SKEW_PACKETS")
    return cx


def _cells(n=20000):
    return workloads.ball(n=n, seed=2111, gamma0=1e-3)


def _timeout(fn):
    with pytest.raises(sgp.SgpError) as e:
        fn()
    assert e.value.code == sgp.ERR_TIMEOUT


def test_forest_solve_alone(skewed):
    c = _cells()
    s = GpuSystem(skewed, c)
    b = dev_tensor(c.forces())
    x = skewed.tree_apply(s.Fac, b)
    torch.cuda.synchronize()
    assert torch.isnan(x).any()
    _timeout(lambda: skewed.tree_apply(s.Fac, b))
    # the same factor in a context that waits
    y = sgp.Context(0).tree_apply(s.Fac, b)
    assert torch.isfinite(y).all()


@pytest.mark.parametrize("precision", [sgp.PREC_F64, sgp.PREC_MIXED])
def test_solves(skewed, precision):
    c = _cells()
    s = GpuSystem(skewed, c, precision=precision)
    F = dev_tensor(c.forces())
    _timeout(lambda: skewed.pcg_solve(s.M, s.Fac, F, precision=precision))
    _timeout(lambda: skewed.pcg_solve(s.M, None, F, precision=precision, precond=sgp.PRECOND_BLOCK_JACOBI))
    v, info = sgp.Context(0).pcg_solve(s.M, s.Fac, F, precision=precision)
    assert info.status == 0


@pytest.mark.parametrize("precision", [sgp.PREC_F64, sgp.PREC_MIXED])
def test_batch(skewed, precision):
    b = GpuBatch(skewed, [3000, 2500], precision=precision)
    _timeout(lambda: skewed.pcg_solve_batched(b.M, b.Fh, b.off, dev_tensor(b.F), precision=precision))


def test_forest_solves_inside_other_calls(skewed):
    """The multi-launch solve (graphs of the forest's launch), a batch cut
    otherwise than its graph, the network."""
    c = _cells()
    s = GpuSystem(skewed, c)
    F = dev_tensor(c.forces())
    net = skewed.mpnn_create((0.1 * np.random.default_rng(1).standard_normal(sgp.MPNN_PARAMS)).astype(np.float32))
    skewed.mpnn_forward(net, s.M, s.Fac, F)
    _timeout(lambda: skewed.mpnn_backward(net, F, sgp.MPNN_LOSS_L2))
    _timeout(lambda: skewed.warm_start(net, s.M, s.Fac, F))
    aug = skewed.augment_tree(s.M, s.T)
    _timeout(lambda: skewed.fcg_solve(s.M, aug, s.Fac, F))
