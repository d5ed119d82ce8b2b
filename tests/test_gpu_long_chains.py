"""Trees whose edges rise or fall along a path, so that a contraction links all vertices in one chain: the
closed form of the result, in a time of the order that random weights take (a chain followed link by link takes
100 times as long)."""
import time

import numpy as np
import pytest

import paper_2104_01126_gb300 as wm
from gpu_common import require_gpu, torch

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
