"""Construction of the search tree, through the EMST it serves, against the oracle bit for bit: sizes
around the block's share (512 and 1024 points), a level's work unit (512 to 2048) and several levels, every
row width, both layouts and types, and nodes whose points all fall on one side (split by count) at every
level.
"""
import numpy as np
import pytest

import oracle
import synthdata
import paper_2104_01126_gb300 as wm
from gpu_common import assert_same_tree, require_gpu, to_np, torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    require_gpu()
    wm.load()


def _check(x, **kw):
    got = wm.emst(x if kw.get("layout") != "soa" else np.ascontiguousarray(x.T), **kw)
    assert_same_tree({k: to_np(got[k]) for k in ("u", "v", "w")}, oracle.emst_at_scale(x))


@pytest.mark.parametrize("n", [511, 512, 513, 1023, 1024, 1025, 2047, 2048, 2049, 2500, 4097, 9001])
@pytest.mark.parametrize("d", [3, 7, 8])
def test_sizes_around_blocks_and_units(n, d):
    _check(synthdata.generate("varden", n, d, seed=n))


@pytest.mark.parametrize("layout", ["aos", "soa"])
@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("d", [1, 2, 5])
def test_layouts_and_types(layout, dtype, d):
    _check(synthdata.gaussian_mixture(3000, d, seed=d, dtype=dtype), layout=layout)


@pytest.mark.parametrize("d", [2, 7])
def test_nodes_split_by_count(d):
    # two far points and 2600 equal ones: the equal ones can only be split by count, in the global levels
    # and in the blocks; then equal points in one coordinate, one ulp apart in another
    x = np.full((2602, d), 0.25, np.float32)
    x[0], x[1] = 0.0, 100.0
    _check(x)
    y = np.zeros((2600, d), np.float32)
    y[:, 0] = np.where(np.arange(2600) % 2, np.float32(1.0), np.nextafter(np.float32(1.0), np.float32(2.0)))
    _check(y)


def test_hdbscan_on_every_row_width_at_several_levels():
    for d in (2, 4, 6, 9, 16):
        x = synthdata.gaussian_mixture(3001, d, seed=40 + d)
        got = wm.hdbscan(torch.from_numpy(x).cuda(), min_pts=5)
        ref = oracle.hdbscan_at_scale(x, 5, 0)
        for k in ("u", "v", "w", "cd", "order"):
            assert np.array_equal(to_np(got[k]), ref[k]), (d, k)
