"""The low-degree kernels decide a vertex from the sums of its row by PE when it
touches few foreign PEs and hand it to the sub-warp queue otherwise: vertices
with 0..8 foreign PEs and degrees 1..32, in warp tiles that are staged and in
tiles too long to stage, against the oracle, for every filter and objective,
as single steps (graph kernels) and inside the engine."""
import numpy as np
import pytest

import oracle as O
from paper_2510_12196_gb300 import gpumap as G
from paper_2510_12196_gb300 import inputs as I

from gpu_helpers import make_ctx, oracle_params

pytestmark = pytest.mark.gpu

HIER, DIST = (4, 4, 3), (1, 10, 100)
K = 48


def _graph(centres=352, leaves=K * 40):
    """Centre i: degree and number of foreign PEs vary with i; its neighbours
    are leaves of its own PE and of the following ones (leaf l lies on PE l mod k)."""
    rng = np.random.default_rng(3)
    n = centres + leaves
    pi = np.empty(n, np.int32)
    pi[:centres] = rng.integers(0, K, centres)
    pi[centres:] = np.arange(leaves) % K
    u, v = [], []
    for i in range(centres):
        deg = 32 - i % 3 if i < 64 else 1 + i % 32  # the first two tiles exceed the staging buffer
        foreign = min(i % 9, deg)
        pes = (pi[i] + np.arange(1, foreign + 1)) % K if foreign else np.array([pi[i]])
        if foreign and i % 2:
            pes = np.append(pes, pi[i])
        row = 0
        for j in range(deg):
            row += rng.integers(1, 3) if j >= len(pes) else 0
            u.append(i)
            v.append(centres + int(pes[j % len(pes)]) + K * ((row + j // len(pes)) % 40))
    p = np.unique(np.stack([u, v], 1), axis=0)
    vw = np.ones(n, np.int32)
    vw[:centres] = rng.integers(1, 30, centres)
    return I.csr_from_pairs(n, p[:, 0], p[:, 1], w=rng.integers(1, 10, len(p)), vw=vw), pi


def test_graph_covers_the_bounds():
    g, pi = _graph()
    foreign = [len(set(pi[g.adj[g.xadj[v]:g.xadj[v + 1]]]) - {pi[v]}) for v in range(352)]
    assert set(range(9)) <= set(foreign) and g.degrees()[:352].max() == 32
    span = g.xadj[32:353:32] - g.xadj[:352:32]
    assert span.max() > 512 and span.min() <= 512


@pytest.mark.parametrize("relax", [(0, 1), (1, 2)])
def test_lp_steps(relax):
    g, pi = _graph()
    ctx = make_ctx(g, HIER, DIST, lp_relax_num=relax[0], lp_relax_den=relax[1])
    try:
        G.map_set_mapping(ctx, 0, pi)
        opi, olock = pi.copy(), (np.arange(g.n) % 11 == 0).astype(np.uint8)
        G.map_set_lock(ctx, 0, olock)
        for _ in range(3):
            mv = G.map_lp_step(ctx, 0)
            opi, olock, pp, gn, inx, omv, cnt = O.lp_step(g, HIER, DIST, opi, olock, relax=relax)
            gpp, gg, ginx, gmv = G.map_get_lp_state(ctx, 0)
            assert mv == cnt and np.array_equal(ginx, inx) and np.array_equal(gpp, pp)
            assert np.array_equal(gg, gn) and np.array_equal(gmv, omv)
            assert np.array_equal(G.map_get_mapping(ctx, 0), opi)
    finally:
        G.map_destroy(ctx)


@pytest.mark.parametrize("objective", [0, 1])
@pytest.mark.parametrize("strong", [False, True])
def test_rebalancing_steps(strong, objective):
    g, pi = _graph()
    L = O.lmax(int(g.vw.sum()), K, 0.0)
    ctx = make_ctx(g, HIER, DIST, eps=0.0, reb_objective=objective)
    try:
        G.map_set_mapping(ctx, 0, pi)
        opi = pi.copy()
        for t in range(1, 4):
            mv = G.map_rebalance_step(ctx, 0, strong, t)
            opi, _, _, cnt = O.rebalance(g, HIER, DIST, L, strong, opi, seed=0x5EED0000, level=0, t=t,
                                         objective=objective)
            assert mv == cnt and np.array_equal(G.map_get_mapping(ctx, 0), opi)
    finally:
        G.map_destroy(ctx)


@pytest.mark.parametrize("variant", [{}, {"lp_relax_num": 1, "lp_relax_den": 2, "reb_objective": 1}])
@pytest.mark.parametrize("mode", [{"engine_max_n": 1 << 15}, {"engine_max_n": -1, "grid_engine_max_n": -1}])
@pytest.mark.parametrize("eps", [0.0, 0.45])
def test_refinement(eps, mode, variant):
    g, pi = _graph()
    L = O.lmax(int(g.vw.sum()), K, eps)
    ctx = make_ctx(g, HIER, DIST, eps=eps, **mode, **variant)
    try:
        G.map_set_mapping(ctx, 0, pi)
        J, mx, it = G.map_refine(ctx, 0, 12)
        opi, oJ, omx, oit, okinds, oJs, oWs = O.refine(g, HIER, DIST, L, pi, rounds=12,
                                                       params=oracle_params(**variant))
        kinds, Js, Ws, _ = G.map_get_refine_trace(ctx)
        assert (J, mx, it) == (oJ, omx, oit)
        assert np.array_equal(kinds, okinds) and np.array_equal(Js, oJs) and np.array_equal(Ws, oWs)
        assert np.array_equal(G.map_get_mapping(ctx, 0), opi)
    finally:
        G.map_destroy(ctx)
