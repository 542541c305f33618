"""The FP32 batched kernel has one substitution height: its autotuner times the buckets and
leaves the handle's table, whatever it holds."""
import ctypes

import numpy as np
import pytest

from helpers import to_dev
from paper_2504_13821_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_f32_table_stays():
    import paper_2504_13821_gb300 as trx
    h = trx.Handle(0)
    probs = []
    for k, n in ((40, 5), (100, 30), (200, 10), (400, 64)):
        A, B = inputs.problem("L", "L", k, n, seed=k, dtype=np.float32)
        probs.append(("S", "L", "L", "N", "N", 1.0, to_dev(A, "cuda:0"), to_dev(B, "cuda:0")))
    before = (4, 8, 16) * 4
    lib, arr = trx.load_library(), (ctypes.c_int * 12)(*before)
    assert lib.trx_batched_set_tuning(h.ptr, 4, arr, 12) == 0
    table = trx.batched_autotune(probs, handle=h)
    assert lib.trx_batched_get_tuning(h.ptr, 4, arr, 12) == 0
    assert tuple(arr) == before and [b["sb"] for b in table["buckets"]] == list(before)
    for b in table["buckets"]:
        assert len(set(b["ms"].values())) == 1 and (b["ms"]["4"] > 0) == (b["problems"] > 0)
    h.close()
