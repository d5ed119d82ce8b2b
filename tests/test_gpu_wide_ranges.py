"""FP64 coordinates of very different magnitudes: far outliers, columns far from 0 beside their range, both; the
oracle's trees element by element, and times of the order that even points take (errors of the FP32 copy that follow
the largest coordinate anywhere blur all other points, whose walks then visit everything)."""
import time

import numpy as np
import pytest

import oracle
import paper_2104_01126_gb300 as wm
from gpu_common import assert_same_tree, require_gpu, to_np, torch


def _set(name, n, d, seed=1):
    g = np.random.default_rng(seed)
    if name == "cauchy":
        return g.standard_cauchy((n, d))
    if name == "lognormal":
        return np.exp(4 * g.standard_normal((n, d)))
    x = g.random((n, d))
    if name == "timestamps":   # one column far from 0
        x[:, 0] = 1.6e9 + 1e5 * x[:, 0]
    elif name == "offset":
        x += 1e8
    elif name == "binades":    # either side of powers of two, where the rounding error doubles
        x = np.where(g.random((n, d)) < 0.5, -1, 1) * 2.0 ** g.integers(-40, 40, (n, d)) * (1 + 2.0 ** -22 * g.standard_normal((n, d)))
    elif name == "columns":    # an exact, a constant, a far and a tiny one
        x[:, 0] = g.permutation(n)
        x[:, 1 % d] = 0.1
        x[:, 2 % d] = -3e12 + 1e6 * x[:, 2 % d]
        x[:, 3 % d] *= 1e-30
    elif name == "far cauchy":
        x = 1e7 + g.standard_cauchy((n, d))
    return x


@pytest.mark.gpu
@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("min_pts", [1, 6])
@pytest.mark.parametrize("n,d", [(9, 2), (700, 4), (3_000, 7), (5_003, 3)])
@pytest.mark.parametrize("name", ["cauchy", "lognormal", "timestamps", "offset", "binades", "columns", "far cauchy"])
def test_trees(name, n, d, min_pts, precision):
    require_gpu()
    x = _set(name, n, d)
    if min_pts == 1:
        got, ref = wm.emst(x, precision=precision), oracle.emst_at_scale(x)
    else:
        got, ref = wm.hdbscan(x, min_pts=min_pts, precision=precision), oracle.hdbscan_at_scale(x, min_pts, 0)
        assert np.array_equal(to_np(got["cd"]), ref["cd"])
    assert_same_tree({k: to_np(got[k]) for k in "uvw"}, ref)


@pytest.mark.gpu
def test_batch_far_from_the_origin():
    require_gpu()
    xs = [_set(name, n, 3, seed=n) for n in (50, 400) for name in ("timestamps", "offset", "cauchy")]
    for mp in (1, 5):
        for x, r in zip(xs, wm.batch([(x, mp, 0) for x in xs])):
            ref = oracle.emst(x) if mp == 1 else oracle.hdbscan(x, mp)
            assert all(np.array_equal(to_np(r[k]), ref[k]) for k in "uvw")


@pytest.mark.gpu
@pytest.mark.parametrize("min_pts", [1, 10])
@pytest.mark.parametrize("name", ["cauchy", "lognormal", "timestamps", "offset"])
def test_times(name, min_pts):
    require_gpu()

    def seconds(x):
        t = torch.from_numpy(x).cuda()
        f = (lambda: wm.emst(t)) if min_pts == 1 else (lambda: wm.hdbscan(t, min_pts=min_pts))
        f()
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        f()
        torch.cuda.synchronize()
        return time.perf_counter() - t0
    assert seconds(_set(name, 300_000, 5)) < 20 * seconds(_set("even", 300_000, 5))
