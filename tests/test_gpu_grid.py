"""The grid solve (one persistent launch per PCG run, one part of the
contraction tree per thread block) against the level kernels on the same
systems: graphs whose parts, top and segments take every shape, from one cell
to a hub that thousands of leaves hang on."""
from __future__ import annotations

import numpy as np
import pytest
import torch

import oracle
import paper_2410_04512_gb300 as sgp
import workloads
from gpu_common import GpuSystem, dev_tensor, oracle_system, rel_err, small_cube
from test_gpu_batched import GpuBatch

pytestmark = pytest.mark.gpu


def _cells(name):
    if name == "one":
        return workloads.Cells("one", np.zeros((1, 3)), np.full(1, 0.5), 1, 0.1, 10.0, 0.25)
    if name == "pair":
        return workloads.Cells("pair", np.array([[0.0, 0, 0], [0.7, 0.1, 0]]), np.full(2, 0.5), 1, 0.1, 10.0, 0.25)
    if name == "hub":
        # a large cell whose contacts with 3000 small, mutually separate ones
        # are the whole graph: one receiver of thousands of leaves
        rng = np.random.default_rng(11)
        k = np.arange(3000) + 0.5
        phi, th = np.arccos(1 - 2 * k / 3000), np.pi * (1 + 5 ** 0.5) * k
        u = np.stack([np.cos(th) * np.sin(phi), np.sin(th) * np.sin(phi), np.cos(phi)], 1)
        pos = np.concatenate([np.zeros((1, 3)), 50.0 * u])
        return workloads.Cells("hub", pos, np.concatenate([[49.8], rng.uniform(0.45, 0.55, 3000)]), 3, 0.1, 10.0, 1e-2)
    if name == "chain":
        x = 0.9 * np.arange(20000)
        pos = np.stack([x, 0.02 * np.sin(0.1 * np.arange(20000)), np.zeros(20000)], 1)
        return workloads.Cells("chain", pos, np.full(20000, 0.5), 9, 0.1, 10.0, 1e-2)
    if name == "forest":
        rng = np.random.default_rng(5)
        pos = np.concatenate([rng.uniform(0, 400, size=(3000, 3)), rng.uniform(0, 9, size=(1500, 3)) + 500.0])
        return workloads.Cells("forest", pos, np.full(4500, 0.5), 8, 0.1, 10.0, 1e-2)
    if name == "sheet":
        return workloads.hex_sheet(nx=121, ny=83, seed=3001)
    if name == "cube129":
        return small_cube(129, seed=1300)
    return workloads.ball(n=61003, seed=2110, gamma0=1e-3)


@pytest.mark.parametrize("precision", [sgp.PREC_F64, sgp.PREC_MIXED])
@pytest.mark.parametrize("name", ["one", "pair", "hub", "chain", "forest", "sheet", "cube129", "ball"])
def test_grid_solve_matches_level_kernels(cuda_device, name, precision):
    """Same operator and stopping test: the two differ in the order of sums.
    Both residuals are at most 1e-10 |F|, so the solutions differ by at most
    2e-10 |F| / lambda_min in the norm; lambda_min >= gamma0, and |v| is at
    least |F| / (gamma0 + lambda_max), which the oracle's tests bound by 1e-8
    on these workloads."""
    c = _cells(name)
    F = dev_tensor(c.forces())
    out = []
    for cap in (0, -1):
        cx = sgp.Context(0)
        cx.set_tuning(bin_cap=cap)
        s = GpuSystem(cx, c, precision=precision)
        v, info = cx.pcg_solve(s.M, s.Fac, F, tol=1e-10, precision=precision)
        assert info.status == 0 and info.true_rel_residual <= 1.05e-10
        out.append((v.cpu().numpy(), info))
    assert abs(out[0][1].iterations - out[1][1].iterations) <= max(3, out[1][1].iterations // 20)
    assert rel_err(out[0][0], out[1][0]) <= 1e-8
    # a second solve from the solution stops at once; twice the same bits
    again, _ = cx.pcg_solve(s.M, s.Fac, F, tol=1e-10, precision=precision)
    assert torch.equal(again, v)


@pytest.mark.parametrize("precision", [sgp.PREC_F64, sgp.PREC_MIXED])
@pytest.mark.parametrize("precond", [sgp.PRECOND_BLOCK_JACOBI, sgp.PRECOND_NONE])
@pytest.mark.parametrize("name", ["one", "pair", "hub", "forest", "sheet", "cube129", "ball"])
def test_grid_rows_match_multi_launch(cuda_device, name, precond, precision):
    """The row-wise preconditioners on parts of rows; bound as above."""
    c = _cells(name)
    F = dev_tensor(c.forces())
    out = []
    for cap in (0, -1):
        cx = sgp.Context(0)
        cx.set_tuning(bin_cap=cap)
        s = GpuSystem(cx, c, precision=precision)
        v, info = cx.pcg_solve(s.M, None, F, tol=1e-10, precond=precond, precision=precision)
        assert info.status == 0 and info.true_rel_residual <= 1.05e-10
        out.append((v.cpu().numpy(), info))
    assert abs(out[0][1].iterations - out[1][1].iterations) <= max(3, out[1][1].iterations // 20)
    assert rel_err(out[0][0], out[1][0]) <= 1e-8


@pytest.mark.parametrize("precision", [sgp.PREC_F64, sgp.PREC_MIXED])
@pytest.mark.parametrize("sizes,ends", [([300, 1200, 0, 1, 2500, 700, 2], None), ([300, 1200, 0, 1, 2500, 700, 2], [0, 1, 4, 5, 7]),
                                        ([900, 20], [0, 2]), ([5] * 170, None)])
def test_grid_batched(cuda_device, sizes, ends, precision):
    """A batch on its instances' parts (or, the last, more instances than
    thread blocks) against the level kernels; `ends`: the solve's systems as
    runs of the graph's instances.  Bound as in the first test."""
    out = []
    for cap in (0, -1):
        cx = sgp.Context(0)
        cx.set_tuning(bin_cap=cap)
        b = GpuBatch(cx, sizes, precision=precision)
        off = b.off if ends is None else b.off[np.asarray(ends)]
        v, infos = cx.pcg_solve_batched(b.M, b.Fh, off, dev_tensor(b.F), tol=1e-10, precision=precision)
        assert all(i.status == 0 and i.true_rel_residual <= 1.05e-10 for i in infos)
        out.append((v.cpu().numpy(), infos))
    for s in range(len(off) - 1):
        lo, hi = int(off[s]), int(off[s + 1])
        assert abs(out[0][1][s].iterations - out[1][1][s].iterations) <= max(3, out[1][1][s].iterations // 20)
        if hi > lo:
            assert rel_err(out[0][0][lo:hi], out[1][0][lo:hi]) <= 1e-8


def test_grid_iterates_at_equal_k(cuda_device):
    """FP64 iterates after k = 1, 5, 30 steps agree with the oracle's PCG to
    1e-9, from zero and from a given start (whose product the launch forms)."""
    c = small_cube(3000, seed=1004)
    cx = sgp.Context(0)
    s = GpuSystem(cx, c)
    o = oracle_system(c)
    F = c.forces()
    f = oracle.prim_msf(c.n, o.ij, o.w)
    fac = oracle.tree_ldlt(f, o.blocks, c.gamma0)
    for k in (1, 5, 30):
        v, info = cx.pcg_solve(s.M, s.Fac, dev_tensor(F), tol=1e-300, maxit=k, raise_on_error=False)
        assert info.iterations == k and info.status == sgp.ERR_NO_CONVERGENCE
        r = oracle.pcg(c.n, o.ij, o.blocks, c.gamma0, F, oracle.PRECOND_TREE, fac, fixed_iters=k)
        assert rel_err(v.cpu().numpy(), r.x) <= 1e-9, k
    x0 = np.random.default_rng(2).standard_normal((c.n, 3))
    Fx = F - oracle.matvec(c.n, o.ij, o.blocks, c.gamma0, x0)
    v, _ = cx.pcg_solve(s.M, s.Fac, dev_tensor(F), v=dev_tensor(x0), x0_given=True, tol=1e-300, maxit=5,
                        raise_on_error=False)
    r = oracle.pcg(c.n, o.ij, o.blocks, c.gamma0, Fx, oracle.PRECOND_TREE, fac, fixed_iters=5)
    assert rel_err(v.cpu().numpy(), x0 + r.x) <= 1e-9
