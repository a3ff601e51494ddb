"""Heavy-edge rounds in one cooperative launch against the graph of kernels and
the oracle: sizes at a warp's, a CTA's and the path's bounds, the limit on
shared GPUs (grid_engine_max_n = -1), none, one and many rounds, and levels
whose two-hop stages run."""
import numpy as np
import pytest

import oracle as O
from paper_2510_12196_gb300 import gpumap as G
from paper_2510_12196_gb300 import inputs as I

from gpu_helpers import make_ctx, oracle_params

pytestmark = pytest.mark.gpu


def _check(g, k=4, **over):
    prm = oracle_params(coarsener=1, coarsest_factor=1, **over)
    lmax = O.lmax(int(g.vw.sum()), k, 0.03)
    maps = []
    for extra in ({}, {"grid_engine_max_n": -1}, {"launch_mode": 1}):
        ctx = make_ctx(g, (k,), (3,), coarsener=1, coarsest_factor=1, max_levels=3, **over, **extra)
        try:
            levels = G.map_coarsen(ctx)
            maps.append([G.map_get_level_graph(ctx, l)[4] for l in range(levels - 1)])
        finally:
            G.map_destroy(ctx)
    M = O.match(g, lmax, prm, level=0)[0]
    assert maps[0] and np.array_equal(maps[0][0], M)
    for other in maps[1:]:
        assert len(other) == len(maps[0]) and all(np.array_equal(a, b) for a, b in zip(maps[0], other))


@pytest.mark.parametrize("n", [33, 127, 128, 129, 2048, 2049, 20011])
def test_sizes(n):
    _check(I.rgg2d(n, I.rgg_radius(n, 9), n, wmax=6))


@pytest.mark.parametrize("n", [262143, 262144, 262145])
def test_bound_of_the_path(n):
    _check(I.rgg2d(n, I.rgg_radius(n, 6), 3, wmax=3))


@pytest.mark.parametrize("rounds", [1, 2, 40])
def test_rounds(rounds):
    _check(I.grid2d(70, 61), match_rounds=rounds)


def test_two_hop_stages():
    """Stars (leaves), complete bipartite parts (twins) and isolated vertices."""
    u, v = [], []
    for c in range(20):
        u += [50 * c] * 30
        v += list(range(50 * c + 1, 50 * c + 31))
        for a in range(31, 33):
            u += [50 * c + a] * 14
            v += list(range(50 * c + 34, 50 * c + 48))
    u, v = np.array(u), np.array(v)
    _check(I.csr_from_pairs(1000, u, v))
    _check(I.rmat(11, 4, 0.57, 0.19, 0.19, 3))
