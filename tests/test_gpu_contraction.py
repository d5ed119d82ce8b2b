"""Dendrograms by contraction levels (wm_single_linkage) against the oracle, element by element, on weights
that set the number of levels and the lengths of the chains: a path whose weights rise along it is one
chain of one level; one whose weights are ordered by bit reversal keeps half of its vertices at every
level, so the last levels meet the one-block tail at every size; saw teeth give many chains that end
together.  Sizes lie on both sides of the tail's 2048 vertices, also after one and two halvings.  Weights are
whole numbers, so w * w and its root are exact on both sides."""
import numpy as np
import pytest

import oracle
import paper_2104_01126_gb300 as wm
from gpu_common import require_gpu, to_np


def _weights(kind, m):
    i = np.arange(m)
    if kind == "rising":
        return i + 1
    if kind == "bits":                     # position 1, 3, 5, .. lightest, then 2, 6, 10, ..
        low = (i + 1) & -(i + 1)
        return np.argsort(np.argsort(low * np.int64(m + 1) + i)) + 1
    period = 37                            # saw
    return np.argsort(np.argsort((i % period) * np.int64(m) + i)) + 1


@pytest.mark.gpu
@pytest.mark.parametrize("kind", ["rising", "bits", "saw"])
@pytest.mark.parametrize("n", [2047, 2048, 2049, 4096, 4097, 8193, 100_001])
def test_paths_of_given_weights(kind, n):
    require_gpu()
    rng = np.random.default_rng(n)
    perm = rng.permutation(n).astype(np.int32)
    u, v, w = perm[:-1], perm[1:], _weights(kind, n - 1)
    start = int(rng.integers(0, n))
    ref = oracle.single_linkage(n, u, v, w.astype(np.float64) ** 2, s=start)
    got = wm.single_linkage(n, u, v, w.astype(np.float64), start=start)
    for key in ("left", "right", "size", "order", "height", "reach"):
        assert np.array_equal(to_np(got[key]), ref[key]), key
