"""Levels large enough for four flags per lane (above 2^19 vertices, a size that
is no multiple of four), against the oracle: label propagation with locks, weak
and strong rebalancing; and mappings set and read back on both sides of the
size where they are converted on the device."""
import numpy as np
import pytest

import oracle as O
from paper_2510_12196_gb300 import gpumap as G
from paper_2510_12196_gb300 import inputs as I

from gpu_helpers import make_ctx

pytestmark = pytest.mark.gpu

HIER, DIST = (4, 3, 5), (1, 10, 100)


def test_steps_above_the_bound():
    g = I.grid2d(733, 719)
    assert g.n > 1 << 19 and g.n % 4 == 3
    k = O.num_pes(HIER)
    L = O.lmax(g.n, k, 0.03)
    pi = ((np.arange(g.n) * k) // g.n).astype(np.int32)
    noise = I.random_mapping(g.n, k, 3)
    flip = I.splitmix64(4, np.arange(g.n, dtype=np.uint64)) % np.uint64(9) == 0
    pi[flip] = noise[flip]
    pi[-3:] = (pi[-4] + 1) % k  # the last, partial word has candidates
    lock = (np.arange(g.n) % 13 == 0).astype(np.uint8)
    ctx = make_ctx(g, HIER, DIST)
    try:
        G.map_set_mapping(ctx, 0, pi)
        assert np.array_equal(G.map_get_mapping(ctx, 0), pi)
        G.map_set_lock(ctx, 0, lock)
        opi, olock = pi.copy(), lock.copy()
        for _ in range(2):
            mv = G.map_lp_step(ctx, 0)
            opi, olock, pp, gn, inx, omv, cnt = O.lp_step(g, HIER, DIST, opi, olock)
            gpp, gg, ginx, gmv = G.map_get_lp_state(ctx, 0)
            assert mv == cnt and np.array_equal(ginx, inx) and np.array_equal(gmv, omv)
            assert np.array_equal(gpp, pp) and np.array_equal(gg, gn)
            assert np.array_equal(G.map_get_mapping(ctx, 0), opi)
        opi[: g.n // 2] = np.minimum(opi[: g.n // 2], 7)
        G.map_set_mapping(ctx, 0, opi)
        for strong in (False, True):
            mv = G.map_rebalance_step(ctx, 0, strong, 1)
            opi, _, _, cnt = O.rebalance(g, HIER, DIST, L, strong, opi, seed=0x5EED0000, level=0, t=1)
            assert mv == cnt and np.array_equal(G.map_get_mapping(ctx, 0), opi)
    finally:
        G.map_destroy(ctx)


@pytest.mark.parametrize("hier", [(4, 8), (4, 3, 5)])
@pytest.mark.parametrize("n", [1, 8192, 8193, 30001])
def test_mappings_set_and_read(n, hier):
    g = I.csr_from_pairs(n, np.arange(n - 1), np.arange(1, n))
    k = O.num_pes(hier)
    ctx = make_ctx(g, hier, DIST[:len(hier)])
    try:
        pi = I.random_mapping(n, k, n)
        G.map_set_mapping(ctx, 0, pi)
        assert np.array_equal(G.map_get_mapping(ctx, 0), pi)
        for bad in (-1, k):
            wrong = pi.copy()
            wrong[n // 2] = bad
            with pytest.raises(G.MapError) as e:
                G.map_set_mapping(ctx, 0, wrong)
            assert e.value.status == 1
            assert np.array_equal(G.map_get_mapping(ctx, 0), pi)  # unchanged
        assert G.map_objective(ctx, 0)[0] == O.objective(g, hier, DIST[:len(hier)], pi)[0]
    finally:
        G.map_destroy(ctx)
