"""Rebalancing with long lists, against the oracle: cut-bucket lists on both
sides of the single-CTA bound (4096) whose remainder is found digit by digit,
blocks whose remainder ends exactly on a digit, and strong steps of the engine
on one cluster and over all SMs with short and long mover lists."""
import numpy as np
import pytest

import oracle as O
from paper_2510_12196_gb300 import gpumap as G
from paper_2510_12196_gb300 import inputs as I

from gpu_helpers import make_ctx, oracle_params

pytestmark = pytest.mark.gpu


def _skewed(n, k, share, seed):
    """Every `share`-th vertex on PE 0, the others spread: one block far above the bound."""
    pi = I.random_mapping(n, k, seed)
    pi[::share] = 0
    return pi


@pytest.mark.parametrize("strong", [False, True])
@pytest.mark.parametrize("nx,ny,k,share,vwmax", [(90, 90, 4, 2, 1), (64, 130, 8, 2, 1), (150, 141, 3, 1, 1),
                                                 (181, 181, 6, 2, 3), (257, 256, 48, 4, 1)])
def test_long_cut_lists(nx, ny, k, share, vwmax, strong):
    g = I.grid2d(nx, ny)
    if vwmax > 1:
        g.vw[:] = 1 + np.arange(g.n) % vwmax
    L = O.lmax(int(g.vw.sum()), k, 0.0)
    ctx = make_ctx(g, (k,), (5,), eps=0.0)
    try:
        pi = _skewed(g.n, k, share, nx)
        G.map_set_mapping(ctx, 0, pi)
        opi = pi.copy()
        for t in range(1, 4):
            mv = G.map_rebalance_step(ctx, 0, strong, t)
            opi, _, _, cnt = O.rebalance(g, (k,), (5,), L, strong, opi, seed=0x5EED0000, level=0, t=t)
            assert mv == cnt and np.array_equal(G.map_get_mapping(ctx, 0), opi), t
    finally:
        G.map_destroy(ctx)


@pytest.mark.parametrize("n,share", [(3000, 3), (20011, 2), (40009, 40), (50021, 2)])
@pytest.mark.parametrize("mode", ["engine", "graph"])
@pytest.mark.parametrize("weak_max", [2, 0])  # 0: strong steps at once, with movers beyond the short lists
def test_refinement_with_strong_steps(n, share, weak_max, mode):
    g = I.rgg2d(n, I.rgg_radius(n, 8), 3, wmax=5)
    hier, dist = (4, 8, 6), (1, 10, 100)
    k = O.num_pes(hier)
    L = O.lmax(int(g.vw.sum()), k, 0.0)
    over = {} if mode == "engine" else dict(engine_max_n=-1, grid_engine_max_n=-1)
    ctx = make_ctx(g, hier, dist, eps=0.0, weak_max=weak_max, **over)
    try:
        pi = _skewed(g.n, k, share, 7)
        G.map_set_mapping(ctx, 0, pi)
        J, mx, it = G.map_refine(ctx, 0, 9)
        opi, oJ, omx, oit, okinds, oJs, oWs = O.refine(g, hier, dist, L, pi, rounds=9, params=oracle_params(weak_max=weak_max))
        kinds, Js, Ws, _ = G.map_get_refine_trace(ctx)
        assert 2 in okinds  # strong steps among them
        assert (J, mx, it) == (oJ, omx, oit)
        assert np.array_equal(kinds, okinds) and np.array_equal(Js, oJs) and np.array_equal(Ws, oWs)
        assert np.array_equal(G.map_get_mapping(ctx, 0), opi)
    finally:
        G.map_destroy(ctx)
