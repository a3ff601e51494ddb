"""Steps whose movers crowd into few blocks (whole mappings on one or two PEs,
a star whose leaves follow the hub), so that most lanes of a warp update one
word: block weights, cut lists of thousands of vertices of one block, one flag
and four flags per lane, code spaces with and without the per-CTA sums, vertex
weights whose sums need 31 bits.  Against the oracle's steps."""
import numpy as np
import pytest

import oracle as O
from paper_2510_12196_gb300 import gpumap as G
from paper_2510_12196_gb300 import inputs as I

from gpu_helpers import make_ctx

pytestmark = pytest.mark.gpu


def _star(n):
    return I.csr_from_pairs(n, np.zeros(n - 1, np.int64), np.arange(1, n, dtype=np.int64))


GRAPHS = {
    "grid": lambda: I.grid2d(130, 97),
    "large grid": lambda: I.grid2d(1 << 10, 513),  # four flags per lane
    "star": lambda: _star(30011),
}


@pytest.mark.parametrize("heavy", [False, True])
@pytest.mark.parametrize("hier,dist", [((4, 8), (1, 10)), ((3, 5), (1, 10)), ((16, 16, 32), (1, 10, 100))])
@pytest.mark.parametrize("name", GRAPHS)
def test_steps(name, hier, dist, heavy):
    g = GRAPHS[name]()
    n, k = g.n, int(np.prod(hier))
    if heavy:
        g.vw[:] = 1 + (np.arange(n) * 7919) % ((1 << 31) // n - 1)
    lmax = O.lmax(int(g.vw.sum()), k, 0.03)
    maps = {"one": np.zeros(n, np.int32), "two": (np.arange(n) % 2 * (k // 2)).astype(np.int32),
            "half": np.where(np.arange(n) < n // 2, k - 1, np.arange(n) * k // n).astype(np.int32)}
    ctx = make_ctx(g, hier, dist)
    try:
        for what, pi in maps.items():
            for strong in (False, True):
                G.map_set_mapping(ctx, 0, pi)
                cnt = G.map_rebalance_step(ctx, 0, strong, 1)
                opi, _, _, ocnt = O.rebalance(g, hier, dist, lmax, strong, pi, seed=0x5EED0000, level=0, t=1)
                assert cnt == ocnt, (what, strong)
                assert np.array_equal(G.map_get_mapping(ctx, 0), opi), (what, strong)
            lock = np.zeros(n, np.uint8)
            G.map_set_mapping(ctx, 0, pi)
            G.map_set_lock(ctx, 0, lock)
            assert G.map_lp_step(ctx, 0) == O.lp_step(g, hier, dist, pi, lock)[6]
            out = G.map_get_mapping(ctx, 0)
            block = np.bincount(out, weights=g.vw, minlength=k).astype(np.int64)
            assert np.array_equal(G.map_block_weights(ctx, 0), block)
    finally:
        G.map_destroy(ctx)
