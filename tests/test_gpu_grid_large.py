"""The persistent launch where its parts no longer fit on chip whole: other
parts' rows read from memory, iterates and residuals in memory, packed vectors,
and FP64 factors too large for the solve whose forest solve alone still is one
launch (inside the graphs of the multi-launch solve)."""
from __future__ import annotations

import math

import pytest
import torch

import paper_2410_04512_gb300 as sgp

pytestmark = pytest.mark.gpu


def _ball(n, seed):
    """(positions, radii, forces) of a spheroid at packing fraction 0.6."""
    g = torch.Generator(device="cuda").manual_seed(seed)

    def u(*shape):
        return torch.rand(*shape, generator=g, device="cuda", dtype=torch.float64)

    d = torch.randn(n, 3, generator=g, device="cuda", dtype=torch.float64)
    pos = d / d.norm(dim=1, keepdim=True) * u(n, 1) ** (1 / 3) * (n * 0.12625 / 0.6) ** (1 / 3)
    return pos.contiguous(), 0.45 + 0.1 * u(n), torch.randn(n, 3, generator=g, device="cuda", dtype=torch.float64)


class System:
    def __init__(self, cap, n, precision, seed=2117):
        self.cx = sgp.Context(0)
        self.cx.set_tuning(bin_cap=cap)
        self.pos, radii, self.F = _ball(n, seed)
        self.graph = self.cx.collision_graph(self.pos, radii)
        m = self.graph.edges().shape[0]
        g = torch.Generator(device="cuda").manual_seed(seed + 1)
        self.gam = torch.exp(math.log(0.1) + math.log(100.0) * torch.rand(2, m, generator=g, device="cuda", dtype=torch.float64))
        self.precision = precision
        self.M = self.cx.friction_assemble(self.graph, self.pos, self.gam[0].contiguous(), self.gam[1].contiguous(), 1e-3,
                                           precision)
        self.T = self.cx.max_spanning_tree(self.M)
        self.Fac = self.cx.tree_factor(self.M, self.T)

    def solve(self, **kw):
        self.cx.launch_count(reset=True)
        v, info = self.cx.pcg_solve(self.M, self.Fac, self.F, tol=1e-10, precision=self.precision, **kw)
        assert info.status == 0 and info.true_rel_residual <= 1.05e-10
        return v.clone(), info, self.cx.launch_count()


@pytest.mark.parametrize("precision,n,persistent", [
    (sgp.PREC_F64, 300_007, True), (sgp.PREC_F64, 450_001, True), (sgp.PREC_F64, 550_003, True),
    (sgp.PREC_F64, 602_003, True), (sgp.PREC_F64, 700_001, False),
    (sgp.PREC_MIXED, 300_007, True), (sgp.PREC_MIXED, 700_001, True), (sgp.PREC_MIXED, 1_000_003, True),
    (sgp.PREC_MIXED, 1_100_003, True)])
def test_large_parts(cuda_device, n, precision, persistent):
    """Against the level kernels.  Both residuals are at most 1e-10 |F|, so the
    solutions differ by 2e-10 |F| / lambda_min at most in the norm; |v| is some
    |F| / gamma of the contacts: 1e-8 on these spheroids, as on the smaller
    ones.  Solved again, and with the factor built again (its parts are dealt
    from lists that atomics fill): the same bits."""
    a, b = System(0, n, precision), System(-1, n, precision)
    va, ia, la = a.solve()
    vb, ib, _ = b.solve()
    assert (la <= 100) == persistent
    assert abs(ia.iterations - ib.iterations) <= max(3, ib.iterations // 20)
    assert float((va - vb).norm() / vb.norm()) <= 1e-8
    assert torch.equal(a.solve()[0], va)
    a.cx.tree_factor(a.M, a.T, a.Fac)
    assert torch.equal(a.solve()[0], va)
    # from the solution: the residual that ended the refinement ends it again
    if precision == sgp.PREC_MIXED:
        w, info, _ = a.solve(v=va.clone(), x0_given=True)
        assert info.iterations == 0 and torch.equal(w, va)


@pytest.mark.parametrize("precision", [sgp.PREC_F64, sgp.PREC_MIXED])
@pytest.mark.parametrize("precond", [sgp.PRECOND_BLOCK_JACOBI, sgp.PRECOND_NONE])
def test_large_parts_of_rows(cuda_device, precond, precision):
    """Row-wise, 60 steps of several hundred: FP64 iterates differ by rounding
    (1e-6 of the residual is far above what 60 steps make of it); in MIXED an
    inner run may end a step apart, which leaves the residual within a factor
    of two.  The same bits again."""
    out = []
    for cap in (0, -1):
        s = System(cap, 500_009, precision)
        kw = dict(precond=precond, precision=precision, tol=1e-300, maxit=60, raise_on_error=False)
        v, info = s.cx.pcg_solve(s.M, None, s.F, **kw)
        v = v.clone()
        out.append((v, info.true_rel_residual))
        again, _ = s.cx.pcg_solve(s.M, None, s.F, **kw)
        assert torch.equal(again, v)
    if precision == sgp.PREC_F64:
        assert abs(out[0][1] - out[1][1]) <= 1e-6 * out[1][1]
        assert float((out[0][0] - out[1][0]).norm() / out[1][0].norm()) <= 1e-6
    else:
        assert 0.5 * out[1][1] <= out[0][1] <= 2.0 * out[1][1]


def test_no_layout_where_none_can_fit(cuda_device):
    """Too many cells for the SMs there are: the factor is built without a
    launch for the persistent solve."""
    n = 1_300_021
    counts = []
    for cap in (0, -1):
        s = System(cap, n, sgp.PREC_F64)
        s.cx.launch_count(reset=True)
        s.cx.tree_factor(s.M, s.T, s.Fac)
        counts.append(s.cx.launch_count())
    assert counts[0] == counts[1]
