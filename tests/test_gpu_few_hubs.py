"""Levels whose long rows are few enough for the fused engine, and just not:
rows per CTA, the longest row, and the entries in rows of 33 to 128 at the
bounds of the rule.  The default route, the graph of kernels and (small graphs)
the oracle refine alike."""
import numpy as np
import pytest

import oracle as O
from paper_2510_12196_gb300 import gpumap as G
from paper_2510_12196_gb300 import inputs as I

from gpu_helpers import make_ctx, oracle_params

pytestmark = pytest.mark.gpu


def _graph(n, hubs):
    """A path with hubs: (vertex, neighbours) each, besides the path's."""
    u, v = np.arange(n - 1), np.arange(1, n)
    rng = np.random.default_rng(n + len(hubs))
    for hub, deg in hubs:
        nb = rng.choice(np.setdiff1d(np.arange(n), [hub - 1, hub, hub + 1]), size=deg - 2, replace=False)
        u, v = np.append(u, np.minimum(nb, hub)), np.append(v, np.maximum(nb, hub))
    p = np.unique(np.stack([u, v], 1), axis=0)
    return I.csr_from_pairs(n, p[:, 0], p[:, 1], w=1 + np.arange(len(p)) % 5)


def _refine(g, hier, dist, pi, **over):
    ctx = make_ctx(g, hier, dist, **over)
    try:
        G.map_set_mapping(ctx, 0, pi)
        out = G.map_refine(ctx, 0, -1)
        return out, G.map_get_mapping(ctx, 0)
    finally:
        G.map_destroy(ctx)


SMALL = {
    "one row of 64": (300, [(150, 64)]),
    "one row of 65": (300, [(150, 65)]),
    "two rows of 33": (200, [(20, 33), (150, 33)]),
    "one row of 128": (300, [(150, 128)]),
    "one row of 129": (300, [(150, 129)]),
    "four rows": (900, [(100 * i + 50, 200) for i in range(4)]),
    "five rows": (900, [(100 * i + 50, 200) for i in range(5)]),
    "five rows on two CTAs": (1100, [(100 * i + 50, 200) for i in range(5)]),
}


@pytest.mark.parametrize("reb_objective", [0, 1])
@pytest.mark.parametrize("name", SMALL)
def test_small(name, reb_objective):
    g = _graph(*SMALL[name])
    hier, dist = (4, 3, 5), (1, 10, 100)
    pi = I.random_mapping(g.n, 60, 3)
    (J, mw, it), out = _refine(g, hier, dist, pi, reb_objective=reb_objective)
    prm = oracle_params(reb_objective=reb_objective)
    opi, oJ, omw, oit = O.refine(g, hier, dist, O.lmax(int(g.vw.sum()), 60, 0.03), pi, params=prm)[:4]
    assert (J, mw, it) == (oJ, omw, oit) and np.array_equal(out, opi)


@pytest.mark.parametrize("n,deg", [(9000, 8191), (9000, 8192), (9000, 8193), (40000, 8192)])
def test_longest_row(n, deg):
    g = _graph(n, [(n // 2, deg)])
    assert g.degrees().max() == deg
    pi = I.random_mapping(n, 32, 5)
    a = _refine(g, (4, 8), (1, 10), pi)
    b = _refine(g, (4, 8), (1, 10), pi, engine_max_n=-1, grid_engine_max_n=-1)
    assert a[0] == b[0] and np.array_equal(a[1], b[1])
