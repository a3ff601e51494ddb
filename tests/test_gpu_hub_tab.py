"""Connectivity tables of hub rows on both sides of the bounds of their classes
(a warp, a CTA, chunk tables over CTAs), for machines whose tables are tiny, of
a size that is no multiple of four words and as large as the classes allow, for
every filter and objective, against the oracle."""
import numpy as np
import pytest

import oracle as O
from paper_2510_12196_gb300 import gpumap as G
from paper_2510_12196_gb300 import inputs as I

from gpu_helpers import make_ctx

pytestmark = pytest.mark.gpu

DEGREES = (65, 256, 257, 511, 1022, 1023, 1024, 1025, 4097, 16384, 16385, 20000)
MACHINES = [((3,), (7,)), ((4, 3, 5), (1, 10, 100)), ((4, 16, 16), (1, 10, 100))]


def _hubs(k, seed=7):
    """Four hubs of each degree (no edges among them) over 24000 vertices joined in a cycle, in blocks by id."""
    rng = np.random.default_rng(seed)
    rest, degs = 24000, np.repeat(DEGREES, 4)
    u = [np.arange(rest)]
    v = [(np.arange(rest) + 1) % rest]
    for i, d in enumerate(degs):
        u.append(np.full(d, rest + i))
        v.append(rng.choice(rest, size=d, replace=False))
    u, v = np.concatenate(u), np.concatenate(v)
    n = rest + len(degs)
    p = np.unique(np.stack([np.minimum(u, v), np.maximum(u, v)], 1), axis=0)
    g = I.csr_from_pairs(n, p[:, 0], p[:, 1], w=rng.integers(1, 30, len(p)),
                         vw=rng.integers(1, 4, n).astype(np.int32))
    assert tuple(g.degrees()[rest:]) == tuple(degs)
    pi = ((np.arange(n) * k) // n).astype(np.int32)
    pi[rest:] = np.arange(len(degs)) % min(k, 2)  # the hubs sit in overweight blocks
    pi[: rest // 3] = np.minimum(pi[: rest // 3], 1)
    return g, pi


@pytest.mark.parametrize("hier,dist", MACHINES)
@pytest.mark.parametrize("mid_deg,split_deg", [(64, 0), (255, 2048)])
@pytest.mark.parametrize("relax", [(0, 1), (1, 2)])
def test_lp_steps(hier, dist, mid_deg, split_deg, relax):
    g, pi = _hubs(O.num_pes(hier))
    ctx = make_ctx(g, hier, dist, mid_deg=mid_deg, split_deg=split_deg, lp_relax_num=relax[0], lp_relax_den=relax[1])
    try:
        opi, olock = pi.copy(), (np.arange(g.n) % 5 == 0).astype(np.uint8)
        G.map_set_mapping(ctx, 0, pi)
        G.map_set_lock(ctx, 0, olock)
        for _ in range(2):
            mv = G.map_lp_step(ctx, 0)
            opi, olock, pp, gn, inx, omv, cnt = O.lp_step(g, hier, dist, opi, olock, relax=relax)
            gpp, gg, ginx, gmv = G.map_get_lp_state(ctx, 0)
            assert mv == cnt and np.array_equal(ginx, inx) and np.array_equal(gpp, pp)
            assert np.array_equal(gg, gn) and np.array_equal(gmv, omv)
            assert np.array_equal(G.map_get_mapping(ctx, 0), opi)
    finally:
        G.map_destroy(ctx)


@pytest.mark.parametrize("hier,dist", MACHINES)
@pytest.mark.parametrize("mid_deg,split_deg", [(64, 0), (255, 2048)])
@pytest.mark.parametrize("objective", [0, 1])
def test_rebalancing_steps(hier, dist, mid_deg, split_deg, objective):
    k = O.num_pes(hier)
    g, pi = _hubs(k)
    L = O.lmax(int(g.vw.sum()), k, 0.03)
    ctx = make_ctx(g, hier, dist, mid_deg=mid_deg, split_deg=split_deg, reb_objective=objective)
    try:
        G.map_set_mapping(ctx, 0, pi)
        opi = pi.copy()
        for t, strong in ((1, False), (2, False), (3, True)):
            mv = G.map_rebalance_step(ctx, 0, strong, t)
            opi, _, _, cnt = O.rebalance(g, hier, dist, L, strong, opi, seed=0x5EED0000, level=0, t=t,
                                         objective=objective)
            assert mv == cnt and np.array_equal(G.map_get_mapping(ctx, 0), opi)
    finally:
        G.map_destroy(ctx)
