"""The watchdog bound (fs_set_iteration_bound) on a small lattice, where one launch runs several iterations: a solve of
no more iterations than the bound is answered, as on any other lattice."""

import numpy as np
import pytest

import inputs
from helpers import rel_resid

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["f64", "f32", "f16"])
def test_a_solve_within_the_bound_is_answered(prec):
    import paper_2212_04430_gb300 as pkg
    dims = (4, 4, 4, 4)
    u = inputs.gauge_field(dims, "haar", seed=1000)
    b = inputs.random_spinor(dims, 29, nvec=3)
    ctx = pkg.Context(dims, device=0)
    try:
        ctx.fs_set_gauge(u)
        # A = 104: the off-diagonal part of M-hat is below 16 / A^2 = 0.0015 of it, so one iteration reaches 1e-3
        ctx.set_iteration_bound(4)
        x, st, rc = ctx.shifted_solve(100.0, [0.0], b, prec=prec, tol=1e-3, rhs_tile=3)
    finally:
        ctx.close()
    assert rc == 0
    assert np.isfinite(x).all()
    for k in range(3):
        assert rel_resid(u, x[0, k], b[k], 100.0, 0.0, dims) <= 1.05e-3
