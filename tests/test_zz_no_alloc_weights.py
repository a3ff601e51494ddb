"""map_objective_noalloc: block weights summed by warp and PE before any table
(mappings with whole warps, parts of warps and single vertices on a PE, weights
of up to 31 bits, out-of-range entries), with and without the per-block table,
and entries that lie before the first row, against numpy."""
import numpy as np
import pytest

from paper_2510_12196_gb300 import gpumap as G
from paper_2510_12196_gb300 import inputs as I

pytestmark = pytest.mark.gpu

HIERS = [((4, 8), (1, 10)), ((3, 5, 7), (1, 10, 100)), ((4, 16, 16), (1, 10, 100)), ((15, 30, 15), (1, 10, 100))]


def _reference(xadj, adj, w, vw, pi, hier, dist):
    k = int(np.prod(hier))
    ok = (pi >= 0) & (pi < k)
    src = np.repeat(np.arange(len(vw)), np.diff(xadj))
    dst, wt = adj[xadj[0]:xadj[-1]].astype(np.int64), w[xadj[0]:xadj[-1]].astype(np.int64)
    both = ok[src] & ok[dst]
    p, q = pi[src[both]].astype(np.int64), pi[dst[both]].astype(np.int64)
    D, below = np.zeros_like(p), 1
    for a, d in zip(hier, dist):
        D = np.where(p // below != q // below, d, D)
        below *= a
    block = np.zeros(k, np.int64)
    np.add.at(block, pi[ok], vw[ok].astype(np.int64))
    return [int((D * wt[both]).sum()), int(block.max())]


@pytest.mark.parametrize("hier,dist", HIERS)
@pytest.mark.parametrize("n", [1, 31, 1023, 1025, 40007])
@pytest.mark.parametrize("kind", ["local", "random", "one", "holes"])
def test_block_weights(n, kind, hier, dist):
    import torch
    k = int(np.prod(hier))
    g = I.rgg2d(n, I.rgg_radius(n, 9.0), 5, wmax=9) if n > 31 else I.grid2d(n, 1)
    draw = I.splitmix64(3, np.arange(n, dtype=np.uint64))
    vw = (1 + draw % np.uint64(2**31 - 1)).astype(np.int32)
    pi = {"local": (np.arange(n) * k // n).astype(np.int32), "one": np.full(n, k - 1, np.int32)}.get(
        kind, I.random_mapping(n, k, 7))
    if kind == "holes":
        pi[draw % np.uint64(3) == 0] = -1
        pi[draw % np.uint64(5) == 0] = k
    lead = 5  # entries before the first row
    xadj = g.xadj + lead
    adj = np.concatenate([np.zeros(lead, np.int32), g.adj])
    w = np.concatenate([np.full(lead, 77, np.int32), g.adjw])
    want = _reference(xadj, adj, w, vw, pi, hier, dist)
    dev = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (xadj, adj, w, vw, pi)]
    out = torch.full((2,), -1, dtype=torch.int64, device="cuda")
    G.map_objective_noalloc(*dev[:4], n, dev[4], hier, dist, out)
    assert out.tolist() == want
