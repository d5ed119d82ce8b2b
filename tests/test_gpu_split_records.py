"""wm_split_records: the fields of interleaved records as arrays of their own, bit for bit, for counts on
both sides of the 48 descriptors of one launch and sizes around a block of threads."""
import numpy as np
import pytest

import paper_2104_01126_gb300 as wm
from gpu_common import require_gpu, to_np, torch

FIELDS = ("u", "v", "w", "left", "right", "height", "size")


@pytest.mark.gpu
@pytest.mark.parametrize("count", [1, 48, 49, 97])
@pytest.mark.parametrize("dendro", [False, True])
def test_fields_equal_the_records(count, dendro):
    require_gpu()
    rng = np.random.default_rng(count)
    ms = rng.choice([0, 1, 255, 256, 257, 5000], size=count)
    off = np.concatenate([[0], np.cumsum(ms)])
    e = np.frombuffer(rng.bytes(16 * int(off[-1]) + 16), dtype=wm.EDGE_DTYPE)
    q = np.frombuffer(rng.bytes(24 * int(off[-1]) + 24), dtype=wm.DNODE_DTYPE)
    eb, qb = (torch.from_numpy(x.view(np.uint8).copy()).cuda() for x in (e, q))
    out = wm._split_records([(eb, qb if dendro else None, int(off[j]), int(ms[j])) for j in range(count)], eb.device)
    for j, r in enumerate(out):
        assert tuple(r) == (FIELDS if dendro else FIELDS[:3])
        for f in r:
            want = (e if f in FIELDS[:3] else q)[f][off[j]:off[j + 1]]
            got = to_np(r[f])
            assert got.dtype == want.dtype and got.tobytes() == want.tobytes(), (j, f)


def test_missing_fields_are_refused():
    lib = wm.load()
    row = np.zeros((1, 10), dtype=np.int64)
    assert lib.wm_split_records(row.ctypes.data, 1, None) == 0      # no records, no launch
    row[0, 2] = 1
    assert lib.wm_split_records(row.ctypes.data, 1, None) == -1
    assert lib.wm_split_records(None, 1, None) == -1
    assert lib.wm_split_records(row.ctypes.data, -1, None) == -1
