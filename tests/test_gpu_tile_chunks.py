"""Hops in chunks of 32, 16 and 8 systems (16, 8 and 4 lanes a site, 8, 16 and 32 sites a block) give the bits of a
system by itself, which another kernel computes, also where a chunk is not full, where the last block's sites are partly beyond the lattice, with slots idle and with two chunks
of systems in a tile."""

import numpy as np
import pytest

import inputs
from helpers import rel_resid

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    import paper_2212_04430_gb300 as p
    return p


@pytest.mark.parametrize("dims,prec,nr,bc_t", [((6, 10, 14, 14), "f16", 12, -1), ((6, 10, 14, 14), "f16", 18, 1),
                                               ((6, 10, 14, 14), "bf16", 18, -1), ((6, 10, 14, 14), "f32", 18, -1),
                                               ((12, 12, 12, 12), "f16", 12, -1), ((12, 12, 12, 12), "f32", 12, 1)])
def test_tiles(pkg, dims, prec, nr, bc_t):
    u = inputs.gauge_field(dims, "smooth", seed=71, eps=0.4)
    b = inputs.random_spinor(dims, 72, nvec=12)
    kw = dict(prec=prec, tol=1e-8, link_compress=nr)
    ctx = pkg.Context(dims, bc_t=bc_t, device=0)
    try:
        ctx.fs_set_gauge(u)
        ref, _, rc = ctx.shifted_solve(-0.2, [0.05, 0.4], b[:2], rhs_tile=1, **kw)
        assert rc == 0 and rel_resid(u, ref[1, 1], b[1], -0.2, 0.4, dims, bc_t) < 1.05e-8
        for tile in (4, 8, 13, 16, 20, 24):
            x, st, rc = ctx.shifted_solve(-0.2, [0.05, 0.4], b, rhs_tile=tile, **kw)
            assert rc == 0 and np.array_equal(x[:, :2], ref)
        assert rel_resid(u, x[0, 11], b[11], -0.2, 0.05, dims, bc_t) < 1.05e-8
    finally:
        ctx.close()


@pytest.mark.parametrize("prec", ["f16", "f32"])
def test_clover_tiles(pkg, prec):
    """The same with the clover term (its M-hat has one operand more)."""
    dims = (4, 6, 2, 10)
    u = inputs.gauge_field(dims, "smooth", seed=73, eps=0.4)
    b = inputs.random_spinor(dims, 74, nvec=6)
    kw = dict(prec=prec, tol=1e-8, verify=1)
    ctx = pkg.Context(dims, device=0)
    try:
        ctx.fs_set_gauge(u)
        ctx.fs_set_clover(1.0)
        ref, _, rc = ctx.shifted_solve(0.1, [0.1, 0.4], b[:2], rhs_tile=1, **kw)
        assert rc == 0
        for tile in (4, 8, 12, 20):
            x, st, rc = ctx.shifted_solve(0.1, [0.1, 0.4], b, rhs_tile=tile, **kw)
            assert rc == 0 and all(s["true_resid"] <= 1.05e-8 for s in st) and np.array_equal(x[:, :2], ref)
    finally:
        ctx.close()
