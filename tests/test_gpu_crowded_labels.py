"""Hub rows most of whose entries lie in a few clusters (complete bipartite
parts and hubs over shared leaves on machines of two and three PEs, whose weight
caps let clusters grow large), by every kernel of the hub clustering: entries of
one label are summed by warp before they meet the table.  Every level's clusters
are the oracle's."""
import numpy as np
import pytest

import oracle as O
from paper_2510_12196_gb300 import gpumap as G
from paper_2510_12196_gb300 import inputs as I

from gpu_helpers import make_ctx, oracle_params

pytestmark = pytest.mark.gpu


def _bipartite(n, hubs, deg, seed):
    """`hubs` rows of about deg / 2 to deg entries over the other vertices."""
    rng = np.random.default_rng(seed)
    u, v = [], []
    for h in range(hubs):
        d = int(rng.integers(deg // 2, deg + 1))
        u.append(np.full(d, h))
        v.append(hubs + rng.permutation(n - hubs)[:d])
    p = np.unique(np.stack([np.concatenate(u), np.concatenate(v)], 1), axis=0)
    return I.csr_from_pairs(n, p[:, 0], p[:, 1], w=rng.integers(1, 50, len(p)))


@pytest.mark.parametrize("k", [2, 3])
@pytest.mark.parametrize("n,hubs,deg", [(3000, 40, 300), (4000, 20, 1000), (6000, 10, 2047), (9000, 8, 4090),
                                        (20000, 6, 8190), (20000, 4, 12000)])
def test_levels(n, hubs, deg, k):
    g = _bipartite(n, hubs, deg, n + k)
    prm = oracle_params(coarsest_factor=1)
    cap = O.lmax(int(g.vw.sum()), k, 0.03) // 4
    ctx = make_ctx(g, (k,), (1,), coarsest_factor=1, max_levels=4)
    try:
        levels = G.map_coarsen(ctx)
        assert levels > 1
        cur = g
        for lvl in range(levels - 1):
            M, nc = O.cluster(cur, max(cap, int(cur.vw.max())), prm, level=lvl)
            assert np.array_equal(G.map_get_level_graph(ctx, lvl)[4], M), lvl
            cur = I.Graph(nc, *O.contract(cur, M, nc))
    finally:
        G.map_destroy(ctx)
