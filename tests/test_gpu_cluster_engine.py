"""The one-launch clustering of small levels against the oracle: sizes around a
warp tile, a CTA, the largest cluster and the bound of the path, rows of up to
128 entries, and weight caps that make few, many (ordered by one CTA) and very
many (ranked by all CTAs) requests contested."""
import numpy as np
import pytest

import oracle as O
from paper_2510_12196_gb300 import gpumap as G
from paper_2510_12196_gb300 import inputs as I

from gpu_helpers import make_ctx, oracle_params

pytestmark = pytest.mark.gpu


def _check(g, k, div, **over):
    prm = oracle_params(cluster_cap_div=div, coarsest_factor=1, **over)
    lmax = O.lmax(int(g.vw.sum()), k, 0.03)
    ctx = make_ctx(g, (k,), (3,), cluster_cap_div=div, coarsest_factor=1, max_levels=3, **over)
    try:
        levels = G.map_coarsen(ctx)
        cur = g
        for lvl in range(levels - 1):
            M, nc = O.cluster(cur, max(lmax // div, int(cur.vw.max())), prm, level=lvl)
            assert np.array_equal(G.map_get_level_graph(ctx, lvl)[4], M), lvl
            cur = I.Graph(nc, *O.contract(cur, M, nc))
    finally:
        G.map_destroy(ctx)
    return levels


@pytest.mark.parametrize("n", [5, 31, 32, 33, 1023, 1024, 1025, 8192, 8193, 20011, 32767, 32768, 32769])
def test_sizes(n):
    g = I.rgg2d(n, I.rgg_radius(n, 9), n, wmax=6)
    g.vw[:] = 1 + np.arange(n) % 3
    assert _check(g, 2, 3) > 1


@pytest.mark.parametrize("div", [4, 60, 1000, 4000])
def test_contested_requests(div):
    g = I.grid2d(160, 150)
    g.vw[:] = 1 + (np.arange(g.n) * 7) % 5
    assert _check(g, 2, div) > 1


def test_rows_up_to_a_quarter_of_the_staging_buffer():
    n = 6000
    rng = np.random.default_rng(2)
    u, v = np.arange(n - 1), np.arange(1, n)
    for hub, deg in ((5, 128), (2000, 127), (4000, 33), (5990, 40)):
        nb = rng.choice(np.setdiff1d(np.arange(n), [hub - 1, hub, hub + 1]), size=deg - 2, replace=False)
        u, v = np.append(u, np.minimum(nb, hub)), np.append(v, np.maximum(nb, hub))
    p = np.unique(np.stack([u, v], 1), axis=0)
    g = I.csr_from_pairs(n, p[:, 0], p[:, 1], w=rng.integers(1, 4, len(p)))
    assert g.degrees().max() >= 128
    assert _check(g, 4, 4) > 1


def test_one_iteration_and_none():
    g = I.grid3d(12, 12, 12)
    assert _check(g, 2, 4, cluster_iters=1) > 1
    _check(g, 2, 4, cluster_iters=0)
