"""Validation of the input graph's entries: sound graphs whose rows begin and
end on every side of the runs and groups of entries that a warp reads at once
(runs of hundreds of empty rows, rows longer than a run) are accepted with the
right weight sum, and one wrong entry at such a place is named."""
import numpy as np
import pytest

import oracle as O
from paper_2510_12196_gb300 import gpumap as G
from paper_2510_12196_gb300 import inputs as I

from gpu_helpers import make_ctx

pytestmark = pytest.mark.gpu


def _graph(kind):
    rng = np.random.default_rng(9)
    if kind == "empty rows":  # 40 vertices with edges, 7 to 900 ids without any between them
        ids = np.cumsum(rng.integers(7, 900, 40))
        u, v = np.triu_indices(40, 1)
        return I.csr_from_pairs(int(ids[-1]) + 500, ids[u], ids[v], w=rng.integers(1, 50, len(u)))
    if kind == "hubs":
        return I.rmat(12, 12, 0.57, 0.19, 0.19, 4)
    if kind == "one group":
        return I.csr_from_pairs(32, np.arange(16), np.arange(16) + 16)
    if kind == "one run":
        return I.csr_from_pairs(129, np.arange(128), np.arange(1, 129))
    return I.grid2d(37, 29)


KINDS = ("empty rows", "hubs", "one group", "one run", "grid")


@pytest.mark.parametrize("kind", KINDS)
def test_sound_graphs_are_accepted(kind):
    g = _graph(kind)
    ctx = make_ctx(g, (2, 2), (1, 10))
    try:
        pi = I.random_mapping(g.n, 4, 1)
        G.map_set_mapping(ctx, 0, pi)
        assert G.map_objective(ctx, 0)[0] == O.objective(g, (2, 2), (1, 10), pi)[0]
    finally:
        G.map_destroy(ctx)


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("at", ["first", "group", "run", "last"])
@pytest.mark.parametrize("fault,words", [("range", "out of range"), ("negative", "out of range"),
                                         ("weight", "weight < 1"), ("asymmetric", "reverse edge"),
                                         ("twin", "reverse edge")])
def test_one_wrong_entry_is_named(kind, at, fault, words):
    g = _graph(kind)
    e = {"first": 0, "group": 32, "run": 256, "last": g.m_dir - 1}[at] % g.m_dir
    adj, w = g.adj.copy(), g.adjw.copy()
    if fault == "range":
        adj[e] = g.n
    elif fault == "negative":
        adj[e] = -1
    elif fault == "weight":
        w[e] = 0
    elif fault == "asymmetric":
        w[e] += 1
    else:  # a neighbour that does not name this vertex (or the vertex itself)
        adj[e] = (adj[e] + 1) % g.n
    with pytest.raises(G.MapError) as err:
        make_ctx(I.Graph(g.n, g.xadj, adj, w, g.vw), (2, 2), (1, 10))
    assert err.value.status == 1
    assert words in str(err.value) or fault == "twin"
