"""The contraction kernels (integer products, pairs grouped by their right vector) against the oracle's on the library's
own solutions: blocks, warps and lattices that do not fill one another, one to six left vectors to a right one, one
displacement to the sixteen that a call may ask for, monomial and dense Gamma, links that are not unitary.

Tolerance: a site's sum errs by less than 24 units of 2^-52 of the largest product |L| |W| |R| over it (integers
below 2^60, sums in units of 2^-60 of it, a warp's sum rounded to 2^-52 at worst), the oracle's by less than 100 x 2^-53;
2e-14 of the sum over the sites of those products covers both, with the rounding of the final FP64 sums."""

import numpy as np
import pytest

import inputs
from oracle import dirac as odirac
from oracle import estimators as oest
from oracle import philox

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    import paper_2212_04430_gb300 as p
    return p


def _gamma(pkg, name):
    if name != "dense":
        return pkg.gamma_matrix(name), {"I": np.eye(4), "g3": odirac.GAMMA[2]}[name]
    rng = np.random.default_rng(17)
    g = rng.normal(size=(4, 4)) + 1j * rng.normal(size=(4, 4))
    return g, g


@pytest.mark.parametrize("dims,nshift,plist,gam,stretch", [
    ((2, 2, 2, 2), 1, [1], "g3", 1.0), ((4, 4, 6, 2), 2, list(range(16)), "I", 1.0), ((6, 6, 2, 10), 5, [0, 1, 3], "g3", 1.0),
    ((4, 4, 4, 8), 6, [0, 2], "dense", 1.0), ((2, 4, 4, 10), 3, [4, 5], "g3", 1.1)])
def test_against_the_oracle(pkg, dims, nshift, plist, gam, stretch):
    u = stretch * inputs.gauge_field(dims, "smooth", seed=51, eps=0.4)
    g, go = _gamma(pkg, gam)
    m, shifts, v = 0.3, [0.1 * (k + 1) for k in range(nshift)], int(np.prod(dims))
    kw = dict(prec="f64", tol=1e-10, rhs_tile=2 * nshift)
    ctx = pkg.Context(dims, device=0)
    try:
        ctx.fs_set_gauge(u)
        out = ctx.variance_sample(m, shifts, g, plist, 1, seed=7, job=3, **kw)
        z = philox.z4_noise(v, 7, 3, philox.VARIANCE_SAMPLE_LEVEL, 0).reshape(v, 4, 3)
        g5 = np.array([1, 1, -1, -1])[:, None]
        x, _, rc = ctx.shifted_solve(m, shifts, np.stack([z, g5 * z]), **kw)
        assert rc == 0
    finally:
        ctx.close()

    def near(got, left, right, p):
        big = np.sqrt((np.abs(left) ** 2).sum() * (np.abs(right) ** 2).sum()) * np.abs(go).sum() * stretch ** p
        return abs(got - oest.contract(u, left, right, go, p, dims)) < 2e-14 * big

    for k, p in enumerate(plist):
        for i in range(nshift):
            assert near(out["a"][0, k, i], z, x[i, 0], p)
            for j in range(i, nshift):
                assert near(out["b"][0, k, i, j], g5 * x[i, 1], x[j, 0], p)


@pytest.mark.parametrize("dims,hpe", [((2, 2, 2, 2), 0), ((6, 6, 2, 10), 3), ((4, 4, 6, 2), 4), ((8, 8, 4, 8), 2)])
def test_staged_groups_match_groups_by_themselves(pkg, dims, hpe):
    """Finished systems of many groups go to their columns in one launch; a group by itself gives the same bits."""
    u = inputs.gauge_field(dims, "smooth", seed=61, eps=0.4)
    kw = dict(prec="f32", tol=1e-8, hpe_order=hpe, estimator="split_even")
    ctx = pkg.Context(dims, device=0)
    try:
        ctx.fs_set_gauge(u)
        run = lambda n, tile: ctx.mlmc_level_trace(0.2, [0.05, 0.4, 0.8], pkg.gamma_matrix("g3"), 1, n, seed=5,
                                                   rhs_tile=tile, **kw)
        many, few = run([9, 7, 5], 13), run([2, 2, 2], 2)
        for a, b in zip(many["samples"], few["samples"]):
            assert np.array_equal(a[:2], b)
    finally:
        ctx.close()
