"""The network's features are ratios: forces of any size that doubles hold give
the same coefficients."""
from __future__ import annotations

import numpy as np
import pytest
import torch

import paper_2410_04512_gb300 as sgp
import workloads
from gpu_common import GpuSystem, dev_tensor

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("e", [-525, -515, -300, 300, 490])
def test_output_scales_with_the_forces(cuda_device, e):
    """A power of two scales F and every product of the forest solve exactly.
    The dot products of the fields then scale by its square, down to 1e-313 at
    2^-525, where doubles still have 11 digits; the features are rounded to
    FP32, so a last bit may turn and moves the output by some 1e-7: 1e-5."""
    c = workloads.ball(n=3000, seed=2116, gamma0=1e-3)
    F = dev_tensor(c.forces())
    cx = sgp.Context(0)
    s = GpuSystem(cx, c)
    net = cx.mpnn_create((0.1 * np.random.default_rng(1).standard_normal(sgp.MPNN_PARAMS)).astype(np.float32))
    v = cx.mpnn_forward(net, s.M, s.Fac, F).clone()
    w = cx.mpnn_forward(net, s.M, s.Fac, F * 2.0 ** e) * 2.0 ** -e
    assert torch.isfinite(w).all()
    assert float((w - v).norm() / v.norm()) <= 1e-5
