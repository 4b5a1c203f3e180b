"""MIXED solves of systems whose coefficients lie near the ends of FP32's range:
the sums of the persistent launch are pairs of floats."""
from __future__ import annotations

import pytest

import paper_2410_04512_gb300 as sgp
import workloads
from gpu_common import GpuSystem, dev_tensor

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precond", [sgp.PRECOND_TREE, sgp.PRECOND_BLOCK_JACOBI])
@pytest.mark.parametrize("e", [-112, -80, 80, 112])
def test_scaled_coefficients(cuda_device, e, precond):
    """Gamma times 2^e (1e-34 to 1e34; its FP32 blocks are in range): the
    velocities times 2^-e, in as many iterations (a few percent: the inner
    solves' rounding is that of other magnitudes where sums are split)."""
    c = workloads.ball(n=20011, seed=2118, gamma0=1e-3)
    F = dev_tensor(c.forces())
    cx = sgp.Context(0)
    s = GpuSystem(cx, c, precision=sgp.PREC_MIXED)
    kw = dict(tol=1e-10, precond=precond, precision=sgp.PREC_MIXED)
    v, info = cx.pcg_solve(s.M, s.Fac, F, **kw)
    k = 2.0 ** e
    M = cx.friction_assemble(s.graph, s.pos, s.gp * k, s.gq * k, c.gamma0 * k, sgp.PREC_MIXED)
    Fac = cx.tree_factor(M, cx.max_spanning_tree(M))
    w, i2 = cx.pcg_solve(M, Fac, F, **kw)
    assert i2.status == 0 and i2.true_rel_residual <= 1e-10
    assert abs(i2.iterations - info.iterations) <= max(3, info.iterations // 20)
    # both residuals are at most 1e-10 |F|: bound as for the other solves
    assert float((w * k - v).norm() / v.norm()) <= 1e-8
