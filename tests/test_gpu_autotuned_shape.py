"""The autotuner times the launch shape of the persistent hop only where the solve takes that hop: a small lattice, whose
iterations run in one launch, keeps the default shape; on a larger one the timed shape changes no bit."""

import numpy as np
import pytest

import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,small", [((4, 4, 4, 8), True), ((8, 8, 8, 8), True), ((12, 12, 12, 12), False)])
def test_shape(dims, small):
    import paper_2212_04430_gb300 as pkg
    u = inputs.gauge_field(dims, "smooth", seed=41, eps=0.3)
    g = pkg.gamma_matrix("g3")
    kw = dict(seed=6, job=3, prec="f16", tol=1e-8, link_compress=12)
    got = []
    tile = 0
    for lanes in (0, 1):
        ctx = pkg.Context(dims, device=0)
        try:
            ctx.fs_set_gauge(u)
            got.append(ctx.mlmc_level_trace(-0.2, [0.05, 0.4], g, 1, [24, 24], rhs_tile=tile, lanes=lanes, **kw))
            if not tile:
                tile, depth, blocks = ctx.tuned_shape("f16", 12)
                assert tile in (8, 16, 32, 64)
                if small or tile % 32:
                    assert (depth, blocks) == (0, 0)
                else:
                    assert depth in (0, 3) and blocks in (0, 2)
        finally:
            ctx.close()
    for a, b in zip(got[0]["samples"], got[1]["samples"]):
        assert np.array_equal(a, b)
