"""A factor kept while the matrix is assembled anew (other coefficients, the
same cells): the persistent launch serves it too, with the new matrix's rows
on the factor's parts."""
from __future__ import annotations

import numpy as np
import pytest
import torch

import paper_2410_04512_gb300 as sgp
import workloads
from gpu_common import GpuSystem, dev_tensor, rel_err
from test_gpu_batched import GpuBatch

pytestmark = pytest.mark.gpu


def _again(cx, s, precision, seed):
    """The matrix with every coefficient changed by up to a fifth."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    k = 0.8 + 0.4 * torch.rand(2, s.gp.numel(), generator=g, device="cuda", dtype=torch.float64)
    return cx.friction_assemble(s.graph, s.pos, s.gp * k[0], s.gq * k[1], s.cells.gamma0, precision)


@pytest.mark.parametrize("precision", [sgp.PREC_F64, sgp.PREC_MIXED])
@pytest.mark.parametrize("n", [2500, 20011])
def test_solve_with_a_kept_factor(cuda_device, n, precision):
    """Against the level kernels: both residuals are at most 1e-10 |F|, so the
    solutions differ by 2e-10 |F| / lambda_min, below 1e-8 of the norm on these
    workloads.  A solve in the persistent launch takes some dozen launches,
    the level kernels some dozen per iteration."""
    c = workloads.ball(n=n, seed=2112, gamma0=1e-3)
    F = dev_tensor(c.forces())
    out = []
    for cap in (0, -1):
        cx = sgp.Context(0)
        cx.set_tuning(bin_cap=cap)
        s = GpuSystem(cx, c, precision=precision)
        runs = []
        for seed in (1, 2, 1):   # two matrices in turn: each on its own rows
            M = _again(cx, s, precision, seed)
            cx.launch_count(reset=True)
            v, info = cx.pcg_solve(M, s.Fac, F, tol=1e-10, precision=precision)
            assert info.status == 0 and info.true_rel_residual <= 1.05e-10
            if cap == 0:
                assert cx.launch_count() <= 100
            runs.append((v.cpu().numpy(), info))
        out.append(runs)
    for (a, ia), (b, ib) in zip(*out):
        assert abs(ia.iterations - ib.iterations) <= max(3, ib.iterations // 20)
        assert rel_err(a, b) <= 1e-8
    np.testing.assert_array_equal(out[0][0][0], out[0][2][0])


@pytest.mark.parametrize("precision", [sgp.PREC_F64, sgp.PREC_MIXED])
def test_batch_with_a_kept_factor(cuda_device, precision):
    """Bound as above, per instance."""
    out = []
    for cap in (0, -1):
        cx = sgp.Context(0)
        cx.set_tuning(bin_cap=cap)
        b = GpuBatch(cx, [300, 1200, 0, 2500], precision=precision)
        t = dev_tensor(workloads.gamma_table(0.1, 10.0))
        gp, gq = workloads.pair_gamma_torch(31, b.ij, t, t)   # other coefficients than the factor's
        M = cx.friction_assemble(b.g, b.pos, gp.contiguous(), gq.contiguous(), 1e-2, precision)
        cx.launch_count(reset=True)
        v, infos = cx.pcg_solve_batched(M, b.Fh, b.off, dev_tensor(b.F), tol=1e-10, precision=precision)
        assert all(i.status == 0 and i.true_rel_residual <= 1.05e-10 for i in infos)
        if cap == 0:
            assert cx.launch_count() <= 100
        out.append(v.cpu().numpy())
    for s in range(len(b.off) - 1):
        lo, hi = int(b.off[s]), int(b.off[s + 1])
        if hi > lo:
            assert rel_err(out[0][lo:hi], out[1][lo:hi]) <= 1e-8


@pytest.mark.parametrize("precision", [sgp.PREC_F64, sgp.PREC_MIXED])
@pytest.mark.parametrize("precond", [sgp.PRECOND_BLOCK_JACOBI, sgp.PRECOND_NONE])
def test_rows_are_laid_out_once_per_assembly(cuda_device, precond, precision):
    """The parts of rows of a row-wise solve are kept for the next solve of the
    same assembly (fewer launches, the same bits) and for no other: another
    preconditioner or the same handle assembled anew."""
    c = workloads.ball(n=20011, seed=2113, gamma0=1e-3)
    F = dev_tensor(c.forces())
    cx = sgp.Context(0)
    s = GpuSystem(cx, c, precision=precision, tree=False)

    def solve(ctx, M, pre=precond):
        ctx.launch_count(reset=True)
        v, info = ctx.pcg_solve(M, None, F, tol=1e-10, precond=pre, precision=precision)
        assert info.status == 0
        return v.clone(), ctx.launch_count()

    v1, l1 = solve(cx, s.M)
    v2, l2 = solve(cx, s.M)
    assert l2 < l1 and torch.equal(v1, v2)
    other = sgp.PRECOND_NONE + sgp.PRECOND_BLOCK_JACOBI - precond
    va, _ = solve(cx, s.M, other)
    vb, _ = solve(sgp.Context(0), s.M, other)
    assert torch.equal(va, vb)
    M = cx.friction_assemble(s.graph, s.pos, 1.3 * s.gp, 0.8 * s.gq, c.gamma0, precision, s.M)   # the same handle
    va, _ = solve(cx, M)
    vb, _ = solve(sgp.Context(0), M)
    assert torch.equal(va, vb) and not torch.equal(va, v1)


def test_flexible_solve_lays_out_its_rows_once(cuda_device):
    """P' on the factor's parts: kept for the next flexible solve, built anew
    with the factor or the augmented forest."""
    c = workloads.ball(n=5003, seed=2114, gamma0=1e-3)
    F = dev_tensor(c.forces())
    cx = sgp.Context(0)
    s = GpuSystem(cx, c)
    aug = cx.augment_tree(s.M, s.T)
    out = []
    for k in range(4):
        if k == 2:
            cx.tree_factor(s.M, s.T, s.Fac)
        if k == 3:
            cx.augment_tree(s.M, s.T, 0, aug)
        cx.launch_count(reset=True)
        v, info = cx.fcg_solve(s.M, aug, s.Fac, F, tol=1e-9)
        assert info.status == 0
        out.append((v.clone(), cx.launch_count()))
    assert out[1][1] < out[0][1] == out[2][1] == out[3][1]
    assert all(torch.equal(v, out[0][0]) for v, _ in out)
