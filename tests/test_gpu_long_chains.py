"""Trees whose edges rise or fall along a path, so that a contraction links all vertices in one chain: the
closed form of the result, in a time of the order that random weights take (a chain followed link by link takes
100 times as long)."""
import time

import numpy as np
import pytest

import paper_2104_01126_gb300 as wm
from gpu_common import require_gpu, to_np, torch

N = 1_000_000


def _seconds(f):
    f()
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    r = f()
    torch.cuda.synchronize()
    return time.perf_counter() - t0, r


@pytest.mark.gpu
@pytest.mark.parametrize("weights", ["rising", "tied", "falling"])
def test_single_linkage_of_a_path(weights):
    require_gpu()
    i = np.arange(N - 1)
    w = {"rising": i + 1.0, "tied": np.ones(N - 1), "falling": N - 1.0 - i}[weights]
    usual, _ = _seconds(lambda: wm.single_linkage(N, i, i + 1, np.random.default_rng(1).permutation(N - 1) + 1.0))
    took, r = _seconds(lambda: wm.single_linkage(N, i, i + 1, w))
    assert np.array_equal(r["order"], np.arange(N))
    assert np.array_equal(r["reach"], np.concatenate([[np.inf], w]))
    assert np.array_equal(r["size"], i + 2) and np.array_equal(r["height"], np.sort(w))
    first, rest = (r["left"], r["right"]) if weights != "falling" else (r["right"], r["left"])
    assert np.array_equal(first[1:], N + i[:-1])                        # each merge holds the one before
    assert np.array_equal(rest, i + 1 if weights != "falling" else (N - 2) - i)
    assert took < 20 * usual


@pytest.mark.gpu
@pytest.mark.parametrize("min_pts", [1, 4])
def test_points_whose_gaps_grow(min_pts):
    # every point's nearest neighbour is the one before it: the first round links all of them
    require_gpu()
    x = np.zeros((N, 2))
    x[:, 0] = np.cumsum(np.arange(N))   # gaps 1, 2, ..., N - 1
    p = np.random.default_rng(2).permutation(N)
    t, u = torch.from_numpy(x[p]).cuda(), torch.from_numpy(np.random.default_rng(3).random((N, 2))).cuda()
    run = wm.emst if min_pts == 1 else lambda y, **kw: wm.hdbscan(y, min_pts=min_pts, **kw)
    usual, _ = _seconds(lambda: run(u, precision="fp64"))
    took, r = _seconds(lambda: run(t, precision="fp64"))
    at = np.argsort(p)   # the row of each point along the line
    if min_pts == 1:
        assert np.array_equal(to_np(r["u"]), np.minimum(at[:-1], at[1:]))
        assert np.array_equal(to_np(r["v"]), np.maximum(at[:-1], at[1:]))
        assert np.array_equal(to_np(r["w"]), np.arange(1.0, N))
    else:
        pad = np.concatenate([np.full(3, -np.inf), x[:, 0], np.full(3, np.inf)])
        near = np.abs(np.lib.stride_tricks.sliding_window_view(pad, 7) - x[:, :1])   # three points on either side
        cd = np.partition(near, min_pts - 1, axis=1)[:, min_pts - 1]
        assert np.array_equal(to_np(r["cd"])[at], cd)
    assert took < 20 * usual
