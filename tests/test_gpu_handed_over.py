"""More queries that walk most of the search tree than a round hands over at once: points about the centre of a
sphere of points, up to sizes where the limit on a walk follows the number of points.  Every one is answered
once, whether by its own walk or by one of several scans: the tree is the oracle's, and where the oracle takes
too long that of the pair traversals."""
import numpy as np
import pytest

import oracle
import paper_2104_01126_gb300 as wm
from gpu_common import assert_same_tree, require_gpu, to_np


def _ball_in_sphere(n, inner, d, radius, seed, dtype):
    g = np.random.default_rng(seed)
    x = g.standard_normal((n - inner, d))
    x /= np.linalg.norm(x, axis=1, keepdims=True)
    return g.permutation(np.concatenate([x, radius * g.standard_normal((inner, d))])).astype(dtype)


@pytest.mark.gpu
@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("min_pts", [1, 10])
@pytest.mark.parametrize("n,inner,d,radius,dtype", [(20_011, 2_500, 3, 1e-7, "f8"), (70_001, 1_500, 2, 1e-6, "f4"),
                                                    (70_001, 600, 5, 1e-7, "f8")])
def test_more_than_one_scan(n, inner, d, radius, dtype, min_pts, precision):
    require_gpu()
    x = _ball_in_sphere(n, inner, d, radius, n + d, dtype)
    if min_pts == 1:
        got, ref = wm.emst(x, precision=precision), oracle.emst_at_scale(x)
    else:
        got, ref = wm.hdbscan(x, min_pts=min_pts, precision=precision), oracle.hdbscan_at_scale(x, min_pts, 0)
        assert np.array_equal(to_np(got["cd"]), ref["cd"])
    assert_same_tree({k: to_np(got[k]) for k in "uvw"}, ref)


@pytest.mark.gpu
@pytest.mark.parametrize("n,inner", [(2_100_003, 40), (2_200_001, 700)])
def test_limit_that_follows_the_number_of_points(n, inner):
    require_gpu()
    x = _ball_in_sphere(n, inner, 3, 1e-3, n, "f4")
    got = wm.emst(x, return_stats=True)
    assert got["stats"].getpairs_visits == 0
    with wm.tuning():   # an override: the pair traversals
        ref = wm.emst(x, return_stats=True)
    assert ref["stats"].getpairs_visits > 0
    assert_same_tree({k: to_np(got[k]) for k in "uvw"}, {k: to_np(ref[k]) for k in "uvw"})


@pytest.mark.gpu
@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("min_pts", [1, 10])
@pytest.mark.parametrize("n,d", [(2_047, 3), (2_048, 3), (3_001, 5), (3_072, 8), (3_073, 8), (4_097, 8)])
def test_smallest_sizes_that_hand_over(n, d, min_pts, precision):
    # up to 3072 points the steps behind the search are one block's: they hold back in the same way
    require_gpu()
    x = _ball_in_sphere(n, 40, d, 1e-6, n + d, "f8")
    if min_pts == 1:
        got, ref = wm.emst(x, precision=precision), oracle.emst_at_scale(x)
    else:
        got, ref = wm.hdbscan(x, min_pts=min_pts, precision=precision), oracle.hdbscan_at_scale(x, min_pts, 0)
        assert np.array_equal(to_np(got["cd"]), ref["cd"])
    assert_same_tree({k: to_np(got[k]) for k in "uvw"}, ref)
