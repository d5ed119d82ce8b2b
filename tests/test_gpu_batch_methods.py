"""A batch has one method whatever wm_opts.method asks for among the forms that materialise the WSPD: the joint
problem of many instances holds a pair for every two of them, and its edges must stop at each instance."""
import ctypes

import numpy as np
import pytest

import synthdata
import paper_2104_01126_gb300 as wm
from gpu_common import require_gpu


@pytest.mark.gpu
@pytest.mark.parametrize("min_pts", [0, 5])
@pytest.mark.parametrize("method", ["gfk", "naive", "gantao"])
def test_batch_materialises_no_wspd(method, min_pts):
    require_gpu()
    lib = wm.load()
    xs = [synthdata.uniform(n, 3, seed=n, dtype=np.float32) for n in range(90, 130)]
    outs = [np.zeros(len(x) - 1, wm.EDGE_DTYPE) for x in xs]
    arr = (wm._Instance * len(xs))()
    for a, x, e in zip(arr, xs, outs):
        a.pts, a.n, a.d, a.min_pts, a.out_edges = x.ctypes.data, len(x), 3, min_pts, e.ctypes.data
    st = wm._Stats()
    opts = wm._opts("fp32", None, st, method=method)
    assert lib.wm_batch(arr, len(xs), wm.WM_F32, wm.WM_AOS, ctypes.byref(opts)) == 0
    assert st.wspd_pairs == 0
    for x, e in zip(xs, outs):
        ref = wm.hdbscan(x, min_pts=min_pts) if min_pts else wm.emst(x)
        assert all(np.array_equal(e[k], ref[k]) for k in "uvw")
