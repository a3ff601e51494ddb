"""map_objective_noalloc splits the CSR entries evenly over its blocks: rows
that straddle or fill whole tiles of 2048 entries, runs of empty rows longer
than a tile's row list, adjacency arrays off a 16-byte boundary, and code
spaces on both sides of the per-block weight tables, against numpy."""
import numpy as np
import pytest

from paper_2510_12196_gb300 import gpumap as G
from paper_2510_12196_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _star(n, hub, leaves):
    v = np.setdiff1d(np.arange(n), [hub])[:leaves]
    return I.csr_from_pairs(n, np.minimum(v, hub), np.maximum(v, hub), w=1 + v % 7,
                            vw=(1 + np.arange(n) % 3).astype(np.int32))


def _sparse(n, pairs):
    u, v = np.array(pairs).T
    return I.csr_from_pairs(n, u, v, w=np.arange(1, len(pairs) + 1))


GRAPHS = {
    "pair": lambda: I.grid2d(2, 1),
    "tile": lambda: _star(1025, 512, 1024),          # exactly one tile of entries
    "tile_and_one": lambda: _star(1026, 0, 1025),
    "hub": lambda: _star(9001, 4500, 9000),          # a row over several tiles
    "empty_runs": lambda: _sparse(70001, [(3, 40000), (4, 70000), (2047, 2048), (65000, 65001)]),
    "edgeless": lambda: I.csr_from_pairs(300, np.zeros(0, np.int64), np.zeros(0, np.int64)),
    "rmat": lambda: I.rmat(12, 16, 0.57, 0.19, 0.19, 11),
}


@pytest.mark.parametrize("hier,dist", [((4, 8, 6), (1, 10, 100)), ((4, 16, 16, 4), (1, 10, 100, 1000))])
@pytest.mark.parametrize("name", sorted(GRAPHS))
def test_rows_of_every_shape(name, hier, dist):
    import torch
    g = GRAPHS[name]()
    k = int(np.prod(hier))
    pi = I.random_mapping(g.n, k, 5)
    src, dst = np.repeat(pi.astype(np.int64), np.diff(g.xadj)), pi.astype(np.int64)[g.adj]
    D, below = np.zeros_like(src), 1
    for a, d in zip(hier, dist):
        D = np.where(src // below != dst // below, d, D)
        below *= a
    top = int(np.bincount(pi, weights=g.vw, minlength=k).max())
    for shift in (0, 1):
        adj = torch.zeros(g.m_dir + 1, dtype=torch.int32, device="cuda")
        w = torch.zeros_like(adj)
        adj[shift:shift + g.m_dir] = torch.from_numpy(g.adj).cuda()
        w[shift:shift + g.m_dir] = torch.from_numpy(g.adjw).cuda()
        x, vw, p = (torch.from_numpy(a).cuda() for a in (g.xadj, g.vw, pi))
        out = torch.full((2,), -1, dtype=torch.int64, device="cuda")
        for weights, want in ((w[shift:], int((D * g.adjw).sum())), (None, int(D.sum()))):
            G.map_objective_noalloc(x, adj[shift:], weights, vw, g.n, p, hier, dist, out)
            assert out.tolist() == [want, top]
