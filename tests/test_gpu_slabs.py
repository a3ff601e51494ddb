"""A context's buffers cut from slabs (no allocator in the config) against one
allocation per buffer (the caller's allocator): the same mappings over repeated
runs of one context, which stops growing, within the admission estimate."""
import numpy as np
import pytest

from paper_2510_12196_gb300 import gpumap as G
from paper_2510_12196_gb300 import inputs as I

pytestmark = pytest.mark.gpu

HIER, DIST = (4, 8, 8), (1, 10, 100)

GRAPHS = {
    "no edges": lambda: I.csr_from_pairs(7, np.zeros(0, np.int64), np.zeros(0, np.int64), name="empty7"),
    "small": lambda: I.grid3d(6, 5, 4),
    "rows of hundreds": lambda: I.rmat(14, 8, 0.57, 0.19, 0.19, 21),
    "one slab": lambda: I.rgg2d(60001, I.rgg_radius(60001, 12.0), 22, wmax=10),
    "above the first slab": lambda: I.grid2d(733, 719),
}


@pytest.mark.parametrize("name", GRAPHS)
def test_slabs_equal_single_allocations(name):
    g = GRAPHS[name]()
    runs = {}
    for own in (True, False):
        cfg = G.map_config_default(5)
        keep = None if own else G.torch_allocator(cfg)
        ctx = G.map_create(g.xadj, g.adj if g.m_dir else None, g.adjw if g.m_dir else None, g.vw, g.n, HIER, DIST,
                           0.03, cfg)
        try:
            out, held = [], []
            for _ in range(3):
                pi = np.zeros(g.n, np.int32)
                out.append((G.map_run(ctx, pi), pi))
                held.append(G.map_stats(ctx).device_bytes)
            peak = G.map_stats(ctx).device_bytes_peak
        finally:
            G.map_destroy(ctx)
        del keep
        assert held[1] == held[2]
        assert peak <= G.map_job_estimate_bytes(g.n, g.m_dir, HIER), (name, own, peak)
        runs[own] = out
    for (j1, p1), (j2, p2) in zip(runs[True], runs[False]):
        assert j1 == j2 and np.array_equal(p1, p2)
