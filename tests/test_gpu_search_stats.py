"""Evaluations and time of the nearest-component search describe the same launches."""
import pytest

import synthdata
import paper_2104_01126_gb300 as wm
from gpu_common import require_gpu


@pytest.mark.gpu
@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_exact_searches_are_counted_apart(precision):
    require_gpu()
    # every point of a lattice has more nearest neighbours than its list holds: the exact searches, which are
    # not timed, evaluate at least those
    s = wm.emst(synthdata.unit_grid(10, 4), precision=precision, return_stats=True)["stats"]
    assert s.ms_bccp_dual > 0 and 0 < s.bccp_dual_evals <= s.bccp_evals - 4 * 10_000
    # in general position nearly all of them are the timed search's
    s = wm.emst(synthdata.uniform(20_000, 3, seed=1), precision=precision, return_stats=True)["stats"]
    assert 0.99 * s.bccp_evals < s.bccp_dual_evals <= s.bccp_evals
