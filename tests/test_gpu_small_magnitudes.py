"""Coordinates whose FP32 copies round below the smallest subnormal, against the FP64 oracle, element by
element: the exact FP64 weights decide however little of them the FP32 copy keeps.  (The tree under the key K
is unique, so every comparison is exact.)"""
import numpy as np
import pytest

import oracle
import paper_2104_01126_gb300 as wm
from gpu_common import assert_same_tree, require_gpu, to_np

HDB_KEYS = ("cd", "left", "right", "size", "height", "order", "reach")


def _check(x, min_pts, precision="fp32"):
    require_gpu()
    if min_pts == 1:
        got = wm.emst(x, precision=precision)
        assert_same_tree({k: to_np(got[k]) for k in "uvw"}, oracle.emst_at_scale(x))
        return
    got, ref = wm.hdbscan(x, min_pts=min_pts, start=2, precision=precision), oracle.hdbscan_at_scale(x, min_pts, 2)
    assert_same_tree({k: to_np(got[k]) for k in "uvw"}, ref)
    for k in HDB_KEYS:
        assert np.array_equal(to_np(got[k]), ref[k]), k


@pytest.mark.gpu
@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("min_pts", [1, 5])
@pytest.mark.parametrize("scale", [2.0 ** -125, 1e-40, 1e-46])
def test_fp64_coordinates_below_the_fp32_range(scale, min_pts, precision):
    _check(scale * np.random.default_rng(1).random((700, 3)), min_pts, precision)


@pytest.mark.gpu
@pytest.mark.parametrize("min_pts", [1, 5])
def test_one_cluster_below_the_fp32_range(min_pts):
    # exact FP32 coordinates but for a cluster about the origin that the copies collapse to one point
    g = np.random.default_rng(2)
    x = np.concatenate([(1 + g.random((900, 2))).astype(np.float32), 1e-46 * g.random((40, 2))])   # FP64
    _check(g.permutation(x), min_pts)


@pytest.mark.gpu
@pytest.mark.parametrize("min_pts", [2, 5, 12])
@pytest.mark.parametrize("d,scale", [(2, 1e-21), (3, 3e-22), (3, 1e-22), (7, 1e-22), (7, 3e-23), (7, 1e-23), (16, 3e-23)])
def test_fp32_distances_that_underflow(d, scale, min_pts):
    # FP32 squared differences vanish beside core distances that do not
    _check((scale * np.random.default_rng(d).random((700, d))).astype(np.float32), min_pts)


@pytest.mark.gpu
def test_inexact_copies_of_distances_that_underflow():
    # the same with rounded copies: the cluster's FP64 coordinates lie 1e-30 beside FP32 ones
    x = (1e-22 * np.random.default_rng(4).random((700, 7))).astype(np.float32).astype(np.float64)
    _check(x + 1e-30 * np.random.default_rng(5).random(x.shape), 5)


@pytest.mark.gpu
@pytest.mark.parametrize("d,scale", [(3, 3e-22), (7, 1e-22)])
def test_distances_that_underflow_in_the_pair_traversals(d, scale):
    require_gpu()
    with wm.tuning():   # an override: the pair traversals
        _check((scale * np.random.default_rng(d).random((700, d))).astype(np.float32), 5)
