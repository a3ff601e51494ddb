"""Clustering of hub rows on both sides of every bound of the row classes (a
thread group, a CTA, a CTA of its own, chunks over CTAs), with unit and with
drawn weights, against the oracle: labels and coarse graph of every level.
The first sub-round (all labels distinct) and the later ones are both in."""
import numpy as np
import pytest

import oracle as O
from paper_2510_12196_gb300 import gpumap as G
from paper_2510_12196_gb300 import inputs as I

from gpu_helpers import make_ctx, oracle_params

pytestmark = pytest.mark.gpu

DEGREES = (129, 255, 256, 1023, 1024, 2047, 2048, 4095, 8191, 8192, 8193, 20000)


def _hubs(wmax, seed=5):
    """Hubs of exactly these degrees (no edges among them) over 24000 vertices joined in a cycle."""
    rng = np.random.default_rng(seed)
    rest, hubs = 24000, len(DEGREES)
    u = [np.arange(rest), np.array([0])]
    v = [(np.arange(rest) + 1) % rest, np.array([2])]
    for i, d in enumerate(DEGREES):
        nb = rng.choice(rest, size=d, replace=False)
        u.append(np.full(d, rest + i))
        v.append(nb)
    u, v = np.concatenate(u), np.concatenate(v)
    p = np.unique(np.stack([np.minimum(u, v), np.maximum(u, v)], 1), axis=0)
    g = I.csr_from_pairs(rest + hubs, p[:, 0], p[:, 1], w=rng.integers(1, wmax + 1, len(p)),
                         vw=rng.integers(1, 4, rest + hubs).astype(np.int32))
    assert tuple(g.degrees()[rest:]) == DEGREES
    return g


@pytest.mark.parametrize("mid_deg", [0, 64])
@pytest.mark.parametrize("wmax,div", [(1, 4), (5, 40)])
def test_hub_rows_cluster_as_the_oracle(wmax, div, mid_deg):
    g = _hubs(wmax)
    k = 8
    prm = oracle_params(cluster_cap_div=div)
    lmax = O.lmax(int(g.vw.sum()), k, 0.03)
    ctx = make_ctx(g, (2, 4), (1, 10), cluster_cap_div=div, mid_deg=mid_deg)
    try:
        levels = G.map_coarsen(ctx)
        assert levels > 1
        cur = g
        for lvl in range(levels - 1):
            M, nc = O.cluster(cur, max(lmax // div, int(cur.vw.max())), prm, level=lvl)
            assert np.array_equal(G.map_get_level_graph(ctx, lvl)[4], M), lvl
            cur = I.Graph(nc, *O.contract(cur, M, nc))
            got = G.map_get_level_graph(ctx, lvl + 1, with_M=False)
            for a, b in zip(got, (cur.xadj, cur.adj, cur.adjw, cur.vw)):
                assert np.array_equal(a, b), lvl
    finally:
        G.map_destroy(ctx)
