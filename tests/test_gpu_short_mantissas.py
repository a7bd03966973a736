"""The FP64 operator and contractions on links of few mantissa bits (fields that were stored in single precision), and
contractions with such left vectors: their integers end in 0x80000000 often, the one 32-bit word whose negative does
not fit 32 bits.

Tolerances as for links of full mantissas: 1e-13 of the largest |U| |psi| for the operator (integer sums and the oracle's
FP64 sums), 2e-14 of |L| |R| for a contraction, and for a residual its tolerance and 5%: the rounding of both
residuals, 1e-14 of ||D|| ||x|| / ||b|| < 100 at these masses, is less than that at 1e-10."""

import numpy as np
import pytest

import inputs
from helpers import oracle_D, rel_resid
from oracle import dirac as odirac
from oracle import estimators as oest
from oracle import philox

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    import paper_2212_04430_gb300 as p
    return p


def _links(kind, dims):
    if kind == "odd":  # every entry an odd multiple of 2^-28, the largest of a link between 1/2 and 1
        rng = np.random.default_rng(19)
        k = 2 * rng.integers(-2 ** 26, 2 ** 26, size=(4, int(np.prod(dims)), 9, 2)) + 1
        k[:, :, 4, 0] = 2 ** 27 + 2 * rng.integers(0, 2 ** 26, size=k.shape[:2]) + 1
        u = np.ldexp(k.astype(np.float64), -28)
        return (u[..., 0] + 1j * u[..., 1]).reshape(4, -1, 3, 3)
    return inputs.gauge_field(dims, kind, seed=23, eps=0.4).astype(np.complex64).astype(np.complex128)


@pytest.mark.parametrize("kind", ["haar", "smooth", "odd"])
def test_operator(pkg, kind):
    import torch
    from paper_2212_04430_gb300.fsmlmc import wilson_dslash_noalloc
    dims = (4, 4, 6, 2)
    u = _links(kind, dims)
    psi = inputs.random_spinor(dims, 24, nvec=3)
    psi[1] = psi[1].astype(np.complex64)
    ref = oracle_D(u, psi, -0.4, 0.15, dims)
    ctx = pkg.Context(dims, device=0)
    try:
        ctx.fs_set_gauge(u)
        got = ctx.wilson_dslash(-0.4, 0.15, psi, prec="f64")
    finally:
        ctx.close()
    bound = 1e-13 * np.abs(u).max() * np.abs(psi).max()
    assert np.abs(got - ref).max() < bound
    du, dpsi = (torch.view_as_real(torch.from_numpy(a)).cuda().contiguous() for a in (u, psi))
    out = torch.zeros_like(dpsi)
    assert wilson_dslash_noalloc(dims, -1, -0.4, 0.15, du.data_ptr(), dpsi.data_ptr(), out.data_ptr(), 3) == 0
    assert np.abs(torch.view_as_complex(out.cpu()).numpy() - ref).max() < bound


@pytest.mark.parametrize("dims,prec", [((4, 4, 4, 8), "f64"), ((4, 4, 4, 8), "f16"), ((8, 8, 8, 22), "f16")])
def test_solutions_solve_the_oracles_system(pkg, dims, prec):
    u = _links("smooth", dims)
    b = inputs.random_spinor(dims, 25, nvec=2)
    tol = 1e-10 if prec == "f64" else 1e-9
    ctx = pkg.Context(dims, device=0)
    try:
        ctx.fs_set_gauge(u)
        x, _, rc = ctx.shifted_solve(-0.2, [0.05], b, prec=prec, tol=tol)
        assert rc == 0
    finally:
        ctx.close()
    for k in range(2):
        assert rel_resid(u, x[0, k], b[k], -0.2, 0.05, dims) <= 1.05 * tol


def test_contractions(pkg):
    dims, plist, m, s = (4, 4, 6, 2), [0, 1, 2], 0.3, 0.1
    u = _links("smooth", dims)
    g5, v = np.array([1, 1, -1, -1])[:, None], int(np.prod(dims))
    kw = dict(prec="f64", tol=1e-10, rhs_tile=2)
    ctx = pkg.Context(dims, device=0)
    try:
        ctx.fs_set_gauge(u)
        out = ctx.variance_sample(m, [s], pkg.gamma_matrix("g3"), plist, 1, seed=7, job=3, **kw)
        z = philox.z4_noise(v, 7, 3, philox.VARIANCE_SAMPLE_LEVEL, 0).reshape(v, 4, 3)
        x, _, rc = ctx.shifted_solve(m, [s], np.stack([z, g5 * z]), **kw)
        assert rc == 0
    finally:
        ctx.close()
    for k, p in enumerate(plist):
        for got, left in ((out["a"][0, k, 0], z), (out["b"][0, k, 0, 0], g5 * x[0, 1])):
            big = np.linalg.norm(left) * np.linalg.norm(x[0, 0]) * np.abs(odirac.GAMMA[2]).sum()
            assert abs(got - oest.contract(u, left, x[0, 0], odirac.GAMMA[2], p, dims)) < 2e-14 * big


def test_left_vectors(pkg):
    """Gamma = diag(g): Gamma^dag z has the entries conj(g) i^k, odd multiples of 2^-29 below 1 (60-bit integers)."""
    dims, plist, m, s = (4, 4, 6, 2), [0, 1], 0.3, 0.1
    u = inputs.gauge_field(dims, "smooth", seed=26, eps=0.4)
    rng = np.random.default_rng(27)
    k = 2 * rng.integers(2 ** 27, 2 ** 28, size=8) + 1
    g = np.diag(np.ldexp(k[:4], -29) - 1j * np.ldexp(k[4:], -29))
    v = int(np.prod(dims))
    kw = dict(prec="f64", tol=1e-10, rhs_tile=1)
    ctx = pkg.Context(dims, device=0)
    try:
        ctx.fs_set_gauge(u)
        out = ctx.variance_sample(m, [s], g, plist, 1, seed=7, job=3, **kw)
        z = philox.z4_noise(v, 7, 3, philox.VARIANCE_SAMPLE_LEVEL, 0).reshape(v, 4, 3)
        x, _, rc = ctx.shifted_solve(m, [s], z[None], **kw)
        assert rc == 0
    finally:
        ctx.close()
    for i, p in enumerate(plist):
        big = np.linalg.norm(z) * np.linalg.norm(x[0, 0]) * np.abs(g).sum()
        assert abs(out["a"][0, i, 0] - oest.contract(u, z, x[0, 0], g, p, dims)) < 2e-14 * big
