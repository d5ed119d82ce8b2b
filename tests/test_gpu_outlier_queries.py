"""Queries that would walk the whole search tree on one lane, against the oracle: points near the centre of a
sphere of points (one, and more than the 512 that a round hands to the shared scan), EMST and HDBSCAN*, both
precisions; and FP64 coordinates at offsets on both sides of the line where the FP32 copy is given up."""
import numpy as np
import pytest

import oracle
import paper_2104_01126_gb300 as wm
from gpu_common import assert_same_tree, require_gpu, to_np


def _sphere(n, inner, d, seed):
    g = np.random.default_rng(seed)
    x = g.standard_normal((n, d))
    x /= np.linalg.norm(x, axis=1, keepdims=True)
    return g.permutation(np.concatenate([x, 1e-7 * g.standard_normal((inner, d))]))


def _same(x, min_pts, precision):
    if min_pts == 1:
        got = wm.emst(x, precision=precision)
        assert_same_tree({k: to_np(got[k]) for k in "uvw"}, oracle.emst_at_scale(x))
        return
    got, ref = wm.hdbscan(x, min_pts=min_pts, precision=precision), oracle.hdbscan_at_scale(x, min_pts, 0)
    assert_same_tree({k: to_np(got[k]) for k in "uvw"}, ref)
    assert np.array_equal(to_np(got["cd"]), ref["cd"])


@pytest.mark.gpu
@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("min_pts", [1, 10])
@pytest.mark.parametrize("n,inner,d,dtype", [(8_191, 1, 3, "f8"), (8_192, 1, 2, "f4"), (20_011, 1, 3, "f4"),
                                             (20_011, 1, 5, "f8"), (20_011, 700, 3, "f8")])
def test_points_inside_a_sphere(n, inner, d, dtype, min_pts, precision):
    require_gpu()
    _same(_sphere(n - inner, inner, d, seed=n + d).astype(dtype), min_pts, precision)


@pytest.mark.gpu
@pytest.mark.parametrize("min_pts", [1, 10])
@pytest.mark.parametrize("offset", [0.0, 1e3, 1e4, 1e5, 1e7])
def test_offset_coordinates(offset, min_pts):
    require_gpu()
    x = offset + np.random.default_rng(3).random((6_007, 3))
    _same(x, min_pts, "fp32")
