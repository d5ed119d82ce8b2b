"""The sort of tree edges into K order (through wm_single_linkage) against the oracle: sizes around the
one-block sort's 2048 edges and around tiles of the passes; runs of equal weights of lengths around the
32 edges that are ordered in place; weights that agree in their 32 leading bits once a zero and a huge
weight stretch the range (8 and 256 of them together).  Roots of the oracle's squares are exact."""
import numpy as np
import pytest

import oracle
import paper_2104_01126_gb300 as wm
from gpu_common import require_gpu, to_np


def _weights(kind, m, rng):
    i = np.arange(m)
    if kind.startswith("run"):
        w = (i // int(kind[3:]) + 1).astype(np.float64)
    elif kind == "wide":
        w = 2.0 ** rng.integers(-250, 250, m)
    else:
        w = (2.0 ** int(kind[4:]) + i)
        w[0] = 0.0
        w[-1] = 2.0 ** 500
    return rng.permutation(w)


@pytest.mark.gpu
@pytest.mark.parametrize("kind", ["run1", "run2", "run32", "run33", "run100000", "wide", "near25", "near30"])
@pytest.mark.parametrize("n", [2, 3, 34, 2049, 2050, 4097, 70_001])
def test_edges_in_k_order(kind, n):
    require_gpu()
    rng = np.random.default_rng([n, len(kind)])
    parent = (rng.random(n - 1) * np.arange(1, n)).astype(np.int64)   # a random tree
    perm = rng.permutation(n).astype(np.int32)
    u, v, w = perm[parent], perm[1:], _weights(kind, n - 1, rng)
    ref = oracle.single_linkage(n, u, v, w * w, s=int(perm[0]))
    got = wm.single_linkage(n, u, v, w, start=int(perm[0]))
    for key in ("left", "right", "size", "order", "height", "reach"):
        assert np.array_equal(to_np(got[key]), ref[key]), key
