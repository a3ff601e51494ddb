"""One-launch clustering where most requests are contested (weight caps of a few
vertices) and where one target has more contested requests than the launch
follows (trees whose leaves all want into one cluster): the oracle's clusters,
on one thread-block cluster and over all SMs, in repeated runs too."""
import numpy as np
import pytest

import oracle as O
from paper_2510_12196_gb300 import gpumap as G
from paper_2510_12196_gb300 import inputs as I

from gpu_helpers import make_ctx, oracle_params

pytestmark = pytest.mark.gpu


def _check(g, div, runs=1):
    prm = oracle_params(cluster_cap_div=div, coarsest_factor=1)
    cap = O.lmax(int(g.vw.sum()), 2, 0.03) // div
    ctx = make_ctx(g, (2,), (3,), cluster_cap_div=div, coarsest_factor=1, max_levels=3)
    try:
        for _ in range(runs):
            levels = G.map_coarsen(ctx)
            cur = g
            for lvl in range(levels - 1):
                M, nc = O.cluster(cur, max(cap, int(cur.vw.max())), prm, level=lvl)
                assert np.array_equal(G.map_get_level_graph(ctx, lvl)[4], M), lvl
                cur = I.Graph(nc, *O.contract(cur, M, nc))
    finally:
        G.map_destroy(ctx)
    assert levels > 1


def _trees(count, children, leaves):
    """Trees of depth two side by side, the edges at their roots heavy, the roots on a path."""
    size = 1 + children * (1 + leaves)
    u, v, w = [], [], []
    for c in range(count):
        root = c * size
        if c:
            u.append(root - size), v.append(root), w.append(1)
        for i in range(children):
            child = root + 1 + i * (1 + leaves)
            u.append(root), v.append(child), w.append(50)
            for j in range(leaves):
                u.append(child), v.append(child + 1 + j), w.append(2)
    return I.csr_from_pairs(count * size, np.array(u), np.array(v), w=np.array(w))


@pytest.mark.parametrize("cap", [2, 3, 8])
@pytest.mark.parametrize("nx,ny", [(64, 64), (181, 181), (256, 200)])
def test_tight_caps(nx, ny, cap):
    g = I.grid2d(nx, ny)
    _check(g, O.lmax(g.n, 2, 0.03) // cap)


@pytest.mark.parametrize("count", [1, 5])
@pytest.mark.parametrize("cap", [300, 1500])
def test_chains_beyond_the_launch(count, cap):
    g = _trees(count, 100, 100)
    assert g.degrees().max() <= 128
    _check(g, O.lmax(g.n, 2, 0.03) // cap, runs=2)
