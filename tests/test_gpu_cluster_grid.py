"""Clustering of the levels above one cluster's size by the cooperative launch,
at both ends of its range, with few, many and very many contested requests,
against the oracle and against the graph of kernels (grid_engine_max_n = -1)."""
import numpy as np
import pytest

from paper_2510_12196_gb300 import gpumap as G
from paper_2510_12196_gb300 import inputs as I

from gpu_helpers import make_ctx
from test_gpu_cluster_engine import _check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("over", [{}, {"grid_engine_max_n": -1}])
@pytest.mark.parametrize("n", [32769, 50021, 131071, 131072, 131073])
def test_sizes(n, over):
    g = I.rgg2d(n, I.rgg_radius(n, 9), n, wmax=6)
    g.vw[:] = 1 + np.arange(n) % 3
    assert _check(g, 2, 3, **over) > 1


@pytest.mark.parametrize("div", [4, 600, 4000])
def test_contested_requests(div):
    g = I.grid2d(211, 199)
    g.vw[:] = 1 + (np.arange(g.n) * 7) % 5
    assert _check(g, 2, div) > 1


def test_repeated_runs():
    g = I.rgg2d(60000, I.rgg_radius(60000, 12), 5, wmax=10)
    out = []
    for over in ({}, {"grid_engine_max_n": -1}):
        ctx = make_ctx(g, (4, 8), (1, 10), **over)
        try:
            for _ in range(2):
                pi = np.zeros(g.n, np.int32)
                out.append((G.map_run(ctx, pi), pi))
        finally:
            G.map_destroy(ctx)
    for j, pi in out[1:]:
        assert j == out[0][0] and np.array_equal(pi, out[0][1])


@pytest.mark.parametrize("wmax", [1, 60])
def test_contested_lists_beyond_the_launch(wmax):
    """Nearly every request is contested: the launch leaves the longest lists to the graph of kernels."""
    g = I.grid2d(300, 300)
    g.vw[:] = 1 + (np.arange(g.n) * 11) % wmax
    assert _check(g, 2, 20000) > 1
