"""Solves on small lattices, where one launch runs whole iterations with a cluster of blocks per system: the
smallest lattice, parities that are not whole warps, the largest lattices that it serves in each storage
precision and the next ones (which the tile kernels serve), batches and right-hand sides by themselves.

Tolerance: the solver's last residual is a full FP64 one, so the oracle's may exceed the tolerance by the
rounding of both alone: 1e-13 of ||D|| ||x|| / ||b|| < 1e3 at these masses, far below 5% of 1e-9."""

import numpy as np
import pytest

import inputs
from helpers import rel_resid

pytestmark = pytest.mark.gpu
TOL = 1e-9


@pytest.fixture(scope="module")
def pkg():
    import paper_2212_04430_gb300 as p
    return p


@pytest.mark.parametrize("dims,prec,nr,bc_t", [
    ((2, 2, 2, 2), "f64", 18, -1), ((2, 2, 2, 2), "f16", 12, -1), ((2, 4, 2, 6), "f32", 18, 1),
    ((2, 4, 2, 6), "f64", 18, 1), ((6, 6, 2, 10), "bf16", 18, -1), ((6, 6, 6, 8), "f64", 18, -1),
    ((6, 6, 6, 8), "f32", 12, 1), ((8, 4, 4, 16), "f64", 18, -1), ((4, 6, 6, 16), "f64", 18, -1),
    ((8, 8, 8, 16), "f16", 12, -1), ((8, 8, 8, 16), "f32", 18, -1), ((10, 6, 10, 14), "bf16", 12, -1),
    ((8, 8, 8, 20), "f16", 18, -1), ((10, 6, 10, 14), "f32", 12, -1), ((6, 10, 14, 14), "f16", 12, -1)])
def test_residuals_and_independence_of_the_batch(pkg, dims, prec, nr, bc_t):
    u = inputs.gauge_field(dims, "smooth", seed=41, eps=0.4)
    b = inputs.random_spinor(dims, 42, nvec=3)
    sig = [0.05, 0.4]
    kw = dict(prec=prec, tol=TOL, link_compress=nr)
    ctx = pkg.Context(dims, bc_t=bc_t, device=0)
    try:
        ctx.fs_set_gauge(u)
        x, st, rc = ctx.shifted_solve(-0.2, sig, b, rhs_tile=5, **kw)  # a queue: six systems in a tile of five
        assert rc == 0 and all(s["status"] == 2 for s in st)
        for j, s in enumerate(sig):
            for k in range(3):
                r = rel_resid(u, x[j, k], b[k], -0.2, s, dims, bc_t)
                assert r <= 1.05 * TOL, (j, k, r)
        x1, _, rc = ctx.shifted_solve(-0.2, sig[1:], b[2:], rhs_tile=1, **kw)
        assert rc == 0 and np.array_equal(x1[0, 0], x[1, 2])
    finally:
        ctx.close()


@pytest.mark.parametrize("prec", ["f64", "f32", "f16"])
def test_sources_of_few_entries(pkg, prec):
    """Free field and a point source: the symmetry makes scalar products vanish, which restarts the solve."""
    dims = (4, 4, 4, 8)
    u = inputs.gauge_field(dims, "smooth", seed=1, eps=0.0)
    b = np.zeros((2, int(np.prod(dims)), 4, 3), np.complex128)
    b[0, 0, 0, 0] = 1.0
    b[1, 5::16, 2, 1] = 1.0
    ctx = pkg.Context(dims, device=0)
    try:
        ctx.fs_set_gauge(u)
        x, st, rc = ctx.shifted_solve(-0.1, [0.2], b, prec=prec, tol=TOL, rhs_tile=2)
        assert rc == 0 and all(s["status"] == 2 for s in st)
        for k in range(2):
            assert rel_resid(u, x[0, k], b[k], -0.1, 0.2, dims) <= 1.05 * TOL
    finally:
        ctx.close()
