"""map_get_lp_state on a context that has run no label-propagation step: the
targets are not set, which every form of the call reports as -1, whether the
ids are converted on the host (at most 8192 vertices), on the device, or not at
all (PE counts that are powers of two).  After a step they are the oracle's."""
import numpy as np
import pytest

import oracle as O
from paper_2510_12196_gb300 import gpumap as G
from paper_2510_12196_gb300 import inputs as I

from gpu_helpers import make_ctx

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("hier,dist", [((4, 3, 5), (1, 10, 100)), ((4, 8), (1, 10))])
@pytest.mark.parametrize("nx,ny", [(3, 1), (128, 64), (8193, 1), (117, 97)])
def test_targets_before_the_first_step(hier, dist, nx, ny):
    g = I.grid2d(nx, ny)
    ctx = make_ctx(g, hier, dist)
    try:
        assert np.all(G.map_get_lp_state(ctx, 0)[0] == -1)
        pi = I.random_mapping(g.n, O.num_pes(hier), 5)
        G.map_set_mapping(ctx, 0, pi)
        assert np.all(G.map_get_lp_state(ctx, 0)[0] == -1)
        G.map_lp_step(ctx, 0)
        assert np.array_equal(G.map_get_lp_state(ctx, 0)[0], O.lp_step(g, hier, dist, pi, np.zeros(g.n, np.uint8))[2])
    finally:
        G.map_destroy(ctx)
