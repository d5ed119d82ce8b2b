"""Core distances of the k-NN walk against the oracle, bit for bit: heap sizes from 1 to the limit of
256 (and block shapes from 128 to 32 threads), n equal to minPts, ties around the k-th value that go to
the tie kernel, more tied points than it holds (the full scan), and inexact FP32 copies.
"""
import numpy as np
import pytest

import oracle
import synthdata
import paper_2104_01126_gb300 as wm
from gpu_common import require_gpu, to_np

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    require_gpu()
    wm.load()


def _check(x, min_pts):
    got = wm.hdbscan(np.ascontiguousarray(x), min_pts=min_pts)
    ref = oracle.hdbscan_at_scale(np.ascontiguousarray(x), min_pts, 0)
    assert np.array_equal(to_np(got["cd"]), ref["cd"])
    assert np.array_equal(to_np(got["w"]), ref["w"])   # MST weights form a unique multiset


@pytest.mark.parametrize("min_pts", [1, 2, 3, 31, 32, 50, 84, 85, 128, 185, 256])
@pytest.mark.parametrize("d", [2, 7])
def test_heap_sizes(min_pts, d):
    _check(synthdata.gaussian_mixture(1200, d, seed=min_pts), min_pts)


@pytest.mark.parametrize("n", [1, 2, 5, 9, 40, 256])
def test_min_pts_equal_to_n(n):
    _check(synthdata.uniform(n, 3, seed=n, dtype=np.float32), n)


@pytest.mark.parametrize("min_pts", [4, 10, 40])
@pytest.mark.parametrize("name", ["grid2", "grid4", "copies30", "copies600", "offset"])
def test_ties_around_the_kth_value(name, min_pts):
    g = np.random.default_rng(7)
    x = {"grid2": lambda: synthdata.unit_grid(40, 2), "grid4": lambda: synthdata.unit_grid(6, 4),
         "copies30": lambda: np.repeat(g.random((50, 3)).astype(np.float32), 30, axis=0),
         "copies600": lambda: np.repeat(g.random((3, 2)).astype(np.float32), 600, axis=0),
         "offset": lambda: 1e4 + g.random((2000, 3))}[name]()
    _check(x, min_pts)
