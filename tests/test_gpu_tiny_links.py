"""The FP64 operator on links of any finite magnitude: those whose largest entry is near or below the smallest normal
double, too.

Tolerance: 1e-13 of the largest |U| |psi|, as for unitary links (integer sums against the oracle's FP64 sums); entries
of a link below 2^-1022 are multiples of 2^-1074, which both sides take as they are."""

import numpy as np
import pytest

import inputs
from helpers import oracle_D

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scale", [2.0 ** -950, 2.0 ** -1000, 2.0 ** -1040, 2.0 ** 900])
def test_hops_over_links_of_extreme_magnitude(scale):
    import paper_2212_04430_gb300 as pkg
    dims = (4, 2, 4, 6)
    u = inputs.gauge_field(dims, "haar", seed=71) * scale
    psi = inputs.random_spinor(dims, 72, nvec=2)
    ctx = pkg.Context(dims, device=0)
    try:
        ctx.fs_set_gauge(u)
        up = 2.0 ** -int(np.log2(scale) * 0.9)  # brings the products back to ordinary magnitudes
        # A = 4 + m + sigma = 0: the hops alone
        got, ref = ctx.wilson_dslash(-4.0, 0.0, psi * up), oracle_D(u, psi * up, -4.0, 0.0, dims)
    finally:
        ctx.close()
    assert np.abs(ref).max() > 0 and np.isfinite(ref.view(np.float64)).all()
    assert np.abs(got - ref).max() < 1e-13 * (np.abs(u).max() * up) * np.abs(psi).max()
