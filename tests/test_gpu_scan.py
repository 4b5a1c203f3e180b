"""The scan behind every build (cells, edges, rows, contraction levels) at the
edges of its tiles and of its one-block form: edge lists and forests bit-exact,
the product and the factor on top of them."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
import paper_2410_04512_gb300 as sgp
import workloads
from gpu_common import GpuSystem, dev_tensor, oracle_system, rel_err

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [8191, 8192, 8193, 16383, 16384, 16385, 24577])
def test_builds_at_scan_edges(cuda_device, n):
    """Integers are exact; the product as in test_gpu_product; the factor's
    solve is checked by its residual, at most 64 eps of |P| |x| (1e-12 with
    room for the norms of these systems, below 100)."""
    c = workloads.ball(n=n, seed=2200 + n, gamma0=1e-2)
    s = GpuSystem(sgp.Context(0), c)
    o = oracle_system(c)
    np.testing.assert_array_equal(s.ij.cpu().numpy(), o.ij)
    f = oracle.prim_msf(c.n, o.ij, o.w)
    np.testing.assert_array_equal(s.T.edge_ids().cpu().numpy(), np.sort(f.tree_edges))
    v = np.random.default_rng(n).standard_normal((c.n, 3))
    y = s.ctx.spmv(s.M, dev_tensor(v)).cpu().numpy()
    assert rel_err(y, oracle.matvec(c.n, o.ij, o.blocks, c.gamma0, v)) <= 1e-12
    x = s.ctx.tree_apply(s.Fac, dev_tensor(v)).cpu().numpy()
    e = f.tree_edges
    r = oracle.matvec(c.n, o.ij[e], o.blocks[e], c.gamma0, x) - v
    assert np.abs(r).max() <= 1e-12 * max(np.abs(x).max(), np.abs(v).max())
