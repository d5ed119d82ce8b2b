"""The nearest-component rounds against the FP64 oracle, element by element, where they can go wrong:
sizes around the search tree's buckets (8 points) and the warp, every row width (d = 1..8, and 9 to 16
under HDBSCAN*), ties that overflow a point's list, inexact FP32 copies, trees deeper than the stack in
shared memory.  The tree under the key K is unique, so every comparison is exact.
"""
import numpy as np
import pytest

import oracle
import synthdata
import paper_2104_01126_gb300 as wm
from gpu_common import assert_same_tree, require_gpu, to_np

pytestmark = pytest.mark.gpu

HDB_KEYS = ("cd", "left", "right", "size", "height", "order", "reach")


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    require_gpu()
    wm.load()


def _check_emst(x):
    got = wm.emst(x, return_stats=True)
    assert_same_tree({k: to_np(got[k]) for k in ("u", "v", "w")}, oracle.emst_at_scale(x))
    s = got["stats"]
    assert s.getpairs_visits == 0 and s.bccp_dual_evals > 0   # the rounds finished the tree themselves


def _check_hdb(x, min_pts, start=0):
    got = wm.hdbscan(x, min_pts=min_pts, start=start, return_stats=True)
    assert got["stats"].tie_overflow == 0 and got["stats"].getpairs_visits == 0
    ref = oracle.hdbscan_at_scale(x, min_pts, start)
    assert_same_tree({k: to_np(got[k]) for k in ("u", "v", "w")}, ref)
    for k in HDB_KEYS:
        assert np.array_equal(to_np(got[k]), ref[k]), k


@pytest.mark.parametrize("n", [2, 3, 4, 5, 8, 9, 16, 17, 31, 32, 33, 64, 65, 127, 129, 257, 1025])
@pytest.mark.parametrize("d", [2, 5])
def test_sizes_around_buckets_and_warps(n, d):
    _check_emst(synthdata.uniform(n, d, seed=n, dtype=np.float32))
    _check_hdb(synthdata.uniform(n, d, seed=n + 1, dtype=np.float32), min(n, 4), start=n - 1)


@pytest.mark.parametrize("d", [1, 2, 3, 4, 5, 6, 7, 8, 9, 12, 15, 16])
def test_every_row_width(d):
    x = synthdata.gaussian_mixture(1500, d, seed=d)
    if d <= 8:
        _check_emst(x)
    _check_hdb(x, 10, start=3)


def _sets():
    g = np.random.default_rng(3)
    yield "grid2", synthdata.unit_grid(45, 2)
    yield "grid3", synthdata.unit_grid(13, 3)
    yield "coarse2", (g.integers(0, 60, (4000, 2)) / 60).astype(np.float32)
    yield "coarse5", g.integers(0, 4, (3000, 5)).astype(np.float32)
    yield "copies3", np.repeat(g.random((800, 3)).astype(np.float32), 3, axis=0)
    yield "copies40", np.repeat(g.random((60, 2)).astype(np.float32), 40, axis=0)
    yield "same", np.ones((300, 3))
    yield "offset", 1e4 + g.random((3000, 2))               # FP32 copies far coarser than the distances
    yield "offset5", 1e5 + g.random((1500, 5))
    yield "gaps", np.stack([np.cumsum(np.arange(3000.0)), np.zeros(3000)], 1)[g.permutation(3000)]
    yield "deep", np.stack([1.5 ** np.arange(90.0), -(1.55 ** np.arange(90.0))], 1)


SETS = dict(_sets())


@pytest.mark.parametrize("name", sorted(SETS))
def test_ties_inexact_copies_and_deep_trees(name):
    _check_emst(np.ascontiguousarray(SETS[name]))


@pytest.mark.parametrize("name", ["grid2", "coarse2", "copies3", "gaps", "deep"])
@pytest.mark.parametrize("min_pts", [2, 5])
def test_hdbscan_with_ties_is_the_canonical_tree(name, min_pts):
    _check_hdb(np.ascontiguousarray(SETS[name]), min_pts)


def test_batch_instances_stay_apart():
    # finished instances (one component, no edge below the cap) beside unfinished ones
    g = np.random.default_rng(5)
    inst = [(synthdata.uniform(n, d, seed=10 * n + d, dtype=np.float32), mp, 0)
            for n, d, mp in [(1, 2, 1), (2, 3, 1), (9, 2, 1), (700, 3, 1), (40, 5, 5), (900, 2, 5), (6, 2, 5)]]
    inst.append((np.repeat(g.random((50, 2)).astype(np.float32), 9, axis=0), 1, 0))
    for (x, mp, s), r in zip(inst, wm.batch(inst)):
        ref = oracle.emst(x) if mp <= 1 else oracle.hdbscan(x, mp, s=s)
        for k in ("u", "v", "w") + (HDB_KEYS if mp > 1 else ()):
            assert np.array_equal(to_np(r[k]), ref[k]), k


@pytest.mark.parametrize("name", ["grid2", "coarse5", "copies40", "offset", "offset5", "gaps", "deep"])
def test_plain_form(name):
    # every distance in FP64: no screen error, the same trees, with rounded and exact FP32 rows
    x = np.ascontiguousarray(SETS[name])
    got = wm.emst(x, precision="fp64", return_stats=True)
    assert got["stats"].max_rel_screen_err == 0.0 and got["stats"].getpairs_visits == 0
    assert_same_tree({k: to_np(got[k]) for k in ("u", "v", "w")}, oracle.emst_at_scale(x))
    if name in ("offset5", "gaps"):
        h = wm.hdbscan(x, min_pts=5, precision="fp64", return_stats=True)
        ref = oracle.hdbscan_at_scale(x, 5, 0)
        assert h["stats"].max_rel_screen_err == 0.0
        for k in ("u", "v", "w") + HDB_KEYS:
            assert np.array_equal(to_np(h[k]), ref[k]), k
