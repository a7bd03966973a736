"""The FP64 operator (its products in integer arithmetic) against the oracle at its edges: lattices whose
parity is not a whole number of warps, system counts around the four a warp holds, entries of any
magnitude, links that are not unitary, zeros and non-finite entries.

Tolerance: the integer sums err by less than 16 units of 2^-55 of the largest |U| |psi| of a site's
neighbours, the oracle's FP64 sums by less than 100 x 2^-53 of it; 1e-13 of the largest product on
the lattice covers both."""

import numpy as np
import pytest

import inputs
from helpers import oracle_D

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    import paper_2212_04430_gb300 as p
    return p


def _dslash(pkg, u, dims, psi, bc_t=-1):
    ctx = pkg.Context(dims, bc_t=bc_t, device=0)
    try:
        ctx.fs_set_gauge(u)
        return ctx.wilson_dslash(-0.4, 0.15, psi, prec="f64")
    finally:
        ctx.close()


@pytest.mark.parametrize("dims,nrhs,bc_t", [((2, 2, 2, 2), 1, -1), ((2, 4, 2, 6), 3, 1), ((6, 2, 4, 10), 5, -1),
                                            ((4, 4, 6, 2), 33, -1), ((4, 4, 4, 4), 4, 1)])
@pytest.mark.parametrize("scale", [1.0, 1e-298, 1e250])
def test_shapes_and_magnitudes(pkg, dims, nrhs, bc_t, scale):
    u = inputs.gauge_field(dims, "haar", seed=5)
    psi = inputs.random_spinor(dims, 6, nvec=nrhs)
    got = _dslash(pkg, u, dims, psi * scale, bc_t) / scale
    ref = oracle_D(u, psi, -0.4, 0.15, dims, bc_t)
    # at 1e-298 the inputs keep 2^-1074 / 1e-298 = 5e-26 of themselves: no further error
    assert np.abs(got - ref).max() < 1e-13 * np.abs(psi).max()


def test_uneven_magnitudes_and_non_unitary_links(pkg):
    dims = (4, 6, 4, 4)
    rng = np.random.default_rng(7)
    u = inputs.gauge_field(dims, "haar", seed=8)
    u = u * np.exp(rng.uniform(-20, 5, u.shape[:2]))[..., None, None]
    psi = inputs.random_spinor(dims, 9, nvec=2)
    psi = psi * np.exp(rng.uniform(-60, 3, psi.shape[:2]))[..., None, None]
    psi[:, ::7] = 0.0
    got, ref = _dslash(pkg, u, dims, psi), oracle_D(u, psi, -0.4, 0.15, dims)
    assert np.abs(got - ref).max() < 1e-13 * np.abs(u).max() * np.abs(psi).max()
    # a site of zeros among zeros stays exactly zero
    one = np.zeros_like(psi)
    one[0, 0, 0, 0] = 1.0
    got = _dslash(pkg, u, dims, one)
    assert np.array_equal(got == 0, oracle_D(u, one, -0.4, 0.15, dims) == 0)


def test_non_finite_entries_spread_to_their_neighbours_only(pkg):
    import torch
    from paper_2212_04430_gb300.fsmlmc import wilson_dslash_noalloc
    dims = (4, 4, 4, 4)
    u = torch.view_as_real(torch.from_numpy(inputs.gauge_field(dims, "haar", seed=3))).cuda().contiguous()
    psi = torch.view_as_real(torch.from_numpy(inputs.random_spinor(dims, 4, nvec=5))).cuda().contiguous()
    psi[2, 0, 1, 1, 0] = float("nan")
    psi[3, 0, 1, 1, 0] = float("inf")
    out = torch.zeros_like(psi)
    assert wilson_dslash_noalloc(dims, -1, -0.4, 0.15, u.data_ptr(), psi.data_ptr(), out.data_ptr(), 5) == 0
    torch.cuda.synchronize()
    bad = ~torch.isfinite(out).flatten(2).all(2).cpu()
    near = torch.zeros(256, dtype=torch.bool)
    near[[0, 1, 3, 4, 12, 16, 48, 64, 192]] = True  # the site and its eight neighbours
    assert not bad[[0, 1, 4]].any()
    assert torch.equal(bad[2], near) and torch.equal(bad[3], near)
