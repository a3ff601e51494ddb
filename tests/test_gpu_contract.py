"""The contraction of larger levels (one counting sort over the coarse targets)
against a plain numpy contraction of every level: entry counts around the
bound of the path and its tiles, one and two radix digits, hubs, empty coarse
rows, weights that share the sort word and weights too wide for it."""
import numpy as np
import pytest

from paper_2510_12196_gb300 import gpumap as G
from paper_2510_12196_gb300 import inputs as I

from gpu_helpers import make_ctx

pytestmark = pytest.mark.gpu


def _path(n, extra=0):
    """A path of n vertices: 2 (n - 1) entries; `extra` isolated vertices after it."""
    u = np.arange(n - 1)
    return I.csr_from_pairs(n + extra, u, u + 1, w=1 + u % 5)


def _wide(g, w):
    return I.Graph(g.n, g.xadj, g.adj, g.adjw * np.int32(w), g.vw)


def _one_heavy_edge(g):
    """Weight 2^29 on the edge (0, 1): 30 bits, beside two coarse ids of 18."""
    w = g.adjw.copy()
    w[0] = w[g.xadj[1]] = 1 << 29
    assert g.adj[0] == 1 and g.adj[g.xadj[1]] == 0
    return I.Graph(g.n, g.xadj, g.adj, w, g.vw)


CASES = {
    "at_bound": (lambda: _path(2049), {}),                 # 4096 entries: the other path
    "above_bound": (lambda: _path(2050), {}),
    "one_tile": (lambda: _path(4097), {}),                 # 8192 entries
    "tile_and_two": (lambda: _path(4098, extra=900), {}),
    "isolated": (lambda: _path(6000, extra=30000), {"cluster_cap_div": 64}),
    "rgg": (lambda: I.rgg2d(30011, I.rgg_radius(30011, 12), 5, wmax=10), {}),
    "wide": (lambda: _wide(I.rgg2d(20011, I.rgg_radius(20011, 12), 5, wmax=3), 2000), {}),
    "too_wide": (lambda: _one_heavy_edge(I.grid2d(700, 700)), {"cluster_cap_div": 15000, "max_levels": 2}),
    "rmat": (lambda: I.rmat(14, 16, 0.57, 0.19, 0.19, 9), {}),
    "rmat_match": (lambda: I.rmat(13, 8, 0.57, 0.19, 0.19, 4), {"coarsener": 1}),
    "star": (lambda: I.csr_from_pairs(9000, np.zeros(8999, np.int64), np.arange(1, 9000)), {"coarsener": 1}),
}


@pytest.mark.parametrize("case", sorted(CASES))
def test_levels_equal_numpy_contraction(case):
    make, over = CASES[case]
    g = make()
    ctx = make_ctx(g, (2, 4), (1, 10), **over)
    try:
        for _ in range(2):  # the second run reuses the level buffers
            levels = G.map_coarsen(ctx)
        fine = G.map_get_level_graph(ctx, 0, with_M=levels > 1)
        assert levels > 1
        for lvl in range(levels - 1):
            coarse = G.map_get_level_graph(ctx, lvl + 1, with_M=lvl + 2 < levels)
            xadj, adj, w, vw, M = fine
            nc = len(coarse[3])
            a, b = np.repeat(M, np.diff(xadj)).astype(np.int64), M[adj].astype(np.int64)
            key, pos = np.unique(a[a != b] * nc + b[a != b], return_inverse=True)
            sums = np.bincount(pos, weights=w[a != b], minlength=len(key)).astype(np.int64)
            rows = np.zeros(nc + 1, np.int64)
            np.cumsum(np.bincount(key // nc, minlength=nc), out=rows[1:])
            assert np.array_equal(coarse[0], rows), lvl
            assert np.array_equal(coarse[1], key % nc), lvl
            assert np.array_equal(coarse[2], sums), lvl
            assert np.array_equal(coarse[3], np.bincount(M, weights=vw, minlength=nc).astype(np.int64)), lvl
            fine = coarse
    finally:
        G.map_destroy(ctx)
