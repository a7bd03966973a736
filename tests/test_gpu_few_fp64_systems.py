"""FP64 storage with one to five systems: a warp of the tile layout's hop holds 8 sites of four systems, or beyond 4096
sites 32 of one system and 16 of two, and no bit of a system's result depends on which. Lattices on both sides of that
line, those above with a half volume (5000, 5040) that is no multiple of 32 or of 16.

Tolerance against the oracle: 1e-13 of the largest |psi| for the operator (integer sums and the oracle's FP64 sums), and
for a residual its tolerance and 5% (rounding of both residuals, as for the other solves)."""

import numpy as np
import pytest

import inputs
from helpers import oracle_D, rel_resid

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims", [(2, 6, 2, 2), (8, 8, 8, 16), (10, 10, 10, 10), (6, 10, 14, 12)])
def test_operator(dims):
    import paper_2212_04430_gb300 as pkg
    u = inputs.gauge_field(dims, "smooth", seed=51, eps=0.4)
    psi = inputs.random_spinor(dims, 52, nvec=5)
    ctx = pkg.Context(dims, device=0)
    try:
        ctx.fs_set_gauge(u)
        five = ctx.wilson_dslash(-0.3, 0.1, psi, prec="f64")
        for n in (1, 2, 3, 4):
            assert np.array_equal(ctx.wilson_dslash(-0.3, 0.1, psi[:n], prec="f64"), five[:n]), n
    finally:
        ctx.close()
    ref = oracle_D(u, psi, -0.3, 0.1, dims)
    assert np.abs(five - ref).max() < 1e-13 * np.abs(psi).max()


@pytest.mark.parametrize("csw", [0.0, 1.0])
def test_solves(csw):
    import paper_2212_04430_gb300 as pkg
    dims = (10, 10, 10, 10)
    u = inputs.gauge_field(dims, "smooth", seed=53, eps=0.3)
    b = inputs.random_spinor(dims, 54, nvec=4)
    ctx = pkg.Context(dims, device=0)
    try:
        ctx.fs_set_gauge(u)
        if csw:
            ctx.fs_set_clover(csw)
        x = {}
        for n in (1, 2, 3, 4):
            x[n], _, rc = ctx.shifted_solve(-0.1, [0.05], b[:n], prec="f64", tol=1e-10, rhs_tile=n)
            assert rc == 0
            assert np.array_equal(x[n][0], x[1][0] if n == 1 else np.concatenate([x[n - 1][0], x[n][0, n - 1:]])), n
    finally:
        ctx.close()
    if not csw:
        for k in range(4):
            assert rel_resid(u, x[4][0, k], b[k], -0.1, 0.05, dims) <= 1.05e-10
