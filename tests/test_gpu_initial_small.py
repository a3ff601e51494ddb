"""The one-CTA breadth-first initial mapping (graphs of at most 12,288 vertices)
against the oracle's FIFO search, on both sides of the bound between its short
and its long row variant (16 entries per vertex) and at its largest size:
vertices without edges before, between and after the components, paths, hubs
longer than a warp, dense graphs, frontiers of more vertices than threads, and
graphs of few vertices and so many entries that the whole GPU searches them."""
import numpy as np
import pytest

import oracle as O
from paper_2510_12196_gb300 import gpumap as G
from paper_2510_12196_gb300 import inputs as I

from gpu_helpers import make_ctx

pytestmark = pytest.mark.gpu


def _scattered(n, pairs, seed):
    """The pairs' vertices spread over n ids, so that ids without edges lie all about."""
    rng = np.random.default_rng(seed)
    used = int(pairs.max()) + 1
    ids = rng.permutation(n)[:used]
    p = np.unique(np.sort(ids[pairs], axis=1), axis=0)
    return I.csr_from_pairs(n, p[:, 0], p[:, 1], vw=rng.integers(1, 9, n).astype(np.int32))


def _graph(name):
    if name == "one":
        return I.csr_from_pairs(1, np.zeros(0, np.int64), np.zeros(0, np.int64))
    if name == "no edges":
        return I.csr_from_pairs(100, np.zeros(0, np.int64), np.zeros(0, np.int64))
    if name == "path":
        return _scattered(3000, np.stack([np.arange(2000), np.arange(1, 2001)], 1), 1)
    if name == "pairs":
        return _scattered(5000, np.arange(3000).reshape(-1, 2), 2)
    if name == "star":
        return _scattered(12288, np.stack([np.zeros(9000, np.int64), np.arange(1, 9001)], 1), 3)
    if name == "mesh":
        return I.rgg2d(12288, I.rgg_radius(12288, 8), 4, wmax=10, shuffled=True)
    if name == "short rows":
        return I.erdos_renyi(1000, 0.0155, 5)
    if name == "long rows":
        return I.erdos_renyi(1000, 0.0165, 5)
    if name == "hubs":
        return I.rmat(13, 16, 0.57, 0.19, 0.19, 6)
    if name == "dense":
        return I.erdos_renyi(700, 0.9, 7)
    if name == "many entries":
        return I.rmat(12, 600, 0.45, 0.22, 0.22, 8)
    raise KeyError(name)


@pytest.mark.parametrize("name", ["one", "no edges", "path", "pairs", "star", "mesh", "short rows", "long rows", "hubs",
                                  "dense", "many entries"])
def test_small_initial_mapping(name):
    g = _graph(name)
    assert g.n <= 12288
    if name in ("short rows", "long rows"):
        assert (g.m_dir <= 16 * g.n) == (name == "short rows")
    k = 12
    ctx = make_ctx(g, (4, 3), (1, 10), coarsest_factor=1 << 30)
    try:
        assert G.map_coarsen(ctx) == 1
        G.map_initial(ctx)
        assert np.array_equal(G.map_get_mapping(ctx, 0), O.initial(g, k))
    finally:
        G.map_destroy(ctx)
