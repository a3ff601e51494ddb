"""Label-propagation steps at the sizes where the vertices per warp of the
flagged-vertex kernels change (4, 8, 16, 32 as the level outgrows the resident
warps), under mappings with every vertex and with few vertices flagged: the
oracle's step, and an exact J after refinement."""
import numpy as np
import pytest

import oracle as O
from paper_2510_12196_gb300 import gpumap as G
from paper_2510_12196_gb300 import inputs as I

from gpu_helpers import make_ctx

pytestmark = pytest.mark.gpu

HIER, DIST = (4, 8), (1, 10)


def _sizes():
    import torch
    warps = (torch.cuda.get_device_properties(0).multi_processor_count if torch.cuda.is_available() else 152) * 64
    return [3, 33] + [m * warps + d for m in (4, 8, 16, 32) for d in (0, 1)]


@pytest.mark.parametrize("n", _sizes())
def test_step_and_objective(n):
    ny = next(d for d in range(int(n ** 0.5), 0, -1) if n % d == 0)
    g = I.grid2d(n // ny, ny)
    ctx = make_ctx(g, HIER, DIST)
    try:
        for pi in (I.random_mapping(n, 32, 3), (np.arange(n) * 32 // n).astype(np.int32)):
            opi, _, pp, gn, inx, mv, cnt = O.lp_step(g, HIER, DIST, pi, np.zeros(n, np.uint8))
            G.map_set_mapping(ctx, 0, pi)
            G.map_set_lock(ctx, 0, np.zeros(n, np.uint8))
            assert G.map_lp_step(ctx, 0) == cnt
            assert np.array_equal(G.map_get_lp_state(ctx, 0)[3], mv)
            assert np.array_equal(G.map_get_mapping(ctx, 0), opi)
    finally:
        G.map_destroy(ctx)
    ctx = make_ctx(g, HIER, DIST, engine_max_n=-1, grid_engine_max_n=-1)
    try:
        G.map_set_mapping(ctx, 0, I.random_mapping(n, 32, 3))
        J, mw, _ = G.map_refine(ctx, 0, 4)
        assert G.map_objective(ctx, 0) == (J, mw)
    finally:
        G.map_destroy(ctx)
