"""A coarsening whose cooperative launches give up waiting (a barrier that one
arrival never reaches, about a second each) goes on as a graph of kernels with
the same levels and the same mapping, and the context keeps working."""
import time

import numpy as np
import pytest

from paper_2510_12196_gb300 import gpumap as G
from paper_2510_12196_gb300 import inputs as I

from gpu_helpers import make_ctx

pytestmark = pytest.mark.gpu

GRAPHS = {"rgg": lambda: I.rgg2d(50021, I.rgg_radius(50021, 12.0), 3, wmax=10), "grid": lambda: I.grid2d(201, 180)}


def _run(g, launches, **over):
    """(levels, J, mapping) of two runs of one context, whose first `launches` launches give up."""
    ctx = make_ctx(g, (4, 8), (1, 10), **over)
    out = []
    try:
        G.map_selftest_coarsen_timeout(ctx, launches)
        for _ in range(2):
            pi = np.zeros(g.n, np.int32)
            J = G.map_run(ctx, pi)
            s = G.map_stats(ctx)
            out.append((s.n[:s.levels], J, pi))
    finally:
        G.map_destroy(ctx)
    return out


def _same(a, b):
    for (na, ja, pa), (nb, jb, pb) in zip(a, b):
        assert list(na) == list(nb) and ja == jb and np.array_equal(pa, pb)


@pytest.mark.parametrize("coarsener", [0, 1])
def test_later_runs_do_not_wait_again(coarsener):
    """The level that gave up takes the graph in the next run, which asks for no further launch there."""
    g = GRAPHS["rgg"]()
    ctx = make_ctx(g, (4, 8), (1, 10), coarsener=coarsener)
    try:
        G.map_selftest_coarsen_timeout(ctx, 100)
        times = []
        for _ in range(2):
            t0 = time.perf_counter()
            G.map_coarsen(ctx)
            times.append(time.perf_counter() - t0)
    finally:
        G.map_destroy(ctx)
    assert times[0] > 0.9 and times[1] < 0.5


@pytest.mark.parametrize("name", GRAPHS)
def test_clustering(name):
    g = GRAPHS[name]()
    _same(_run(g, 1), _run(g, 0))


@pytest.mark.parametrize("name", GRAPHS)
def test_matching(name):
    g = GRAPHS[name]()
    _same(_run(g, 2, coarsener=1), _run(g, 0, coarsener=1))
