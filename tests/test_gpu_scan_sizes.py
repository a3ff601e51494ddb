"""Scans on both sides of the one-launch bound (16384 items), seen through the
paths that are built on them: numbering of clusters and coarse rows on levels of
n vertices (scans of n and of 2 n + 1 items), against the oracle."""
import numpy as np
import pytest

from paper_2510_12196_gb300 import inputs as I

from test_gpu_cluster_engine import _check
from test_gpu_match_rounds import _check as _check_matching

pytestmark = pytest.mark.gpu


def _graph(n):
    g = I.rgg2d(n, I.rgg_radius(n, 7), n, wmax=5, shuffled=True)
    g.vw[:] = 1 + np.arange(n) % 4
    return g


@pytest.mark.parametrize("n", [1, 2, 1023, 1024, 1025, 8191, 8192, 15360, 16383, 16384, 16385, 20000])
def test_clustering_levels(n):
    if n < 3:
        g = I.csr_from_pairs(n, np.arange(n - 1), np.arange(1, n))
        _check(g, 2, 2)
    else:
        assert _check(_graph(n), 2, 4) > 1


@pytest.mark.parametrize("n", [1024, 16384, 16385])
@pytest.mark.parametrize("launch_mode", [0, 1])
def test_both_launch_modes(n, launch_mode):
    assert _check(_graph(n), 2, 300, launch_mode=launch_mode) > 1


@pytest.mark.parametrize("n", [16383, 16384, 16385])
def test_matching_levels(n):
    _check_matching(_graph(n))
