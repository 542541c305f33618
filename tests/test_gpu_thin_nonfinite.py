"""Few right-hand sides in FP32 (the thin solves and products, whole calls and leaves) with
an Inf in the right-hand side at any row of a 4-row tile: the rows before it and the other
columns are bitwise those of the call without it, and its own row is an Inf."""
import numpy as np
import pytest

from helpers import to_dev
from paper_2504_13821_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

ROWS = [1, 62, 63, 65, 66, 131, 190, 255]


@pytest.mark.parametrize("op,k,nrhs,option", [
    ("trsm", 900, 20, "OPT_THIN"), ("trmm", 900, 20, "OPT_THIN"), ("trsm", 300, 12, "OPT_THIN"),
    ("trsm", 256, 100, None), ("trsm", 512, 300, None), ("trsm", 1000, 400, None),
    ("trsm", 2048, 600, None), ("trmm", 512, 16, None)])
def test_inf_at_any_row(op, k, nrhs, option):
    import paper_2504_13821_gb300 as trx
    h = trx.Handle(0)
    if option:
        h.set_option(getattr(trx, option), 1)
    A, B = inputs.problem("L", "L", k, nrhs, seed=5, dtype=np.float32)
    At, B0, B1 = (to_dev(z, "cuda:0") for z in (A, B, B))
    rows = ROWS + [k // 2 + 3, k - 3]
    for c, r in enumerate(rows):
        B1[r, c] = float("inf")
    for z in (B0, B1):
        getattr(trx, op)("L", "L", "N", "N", 1.0, At, z, handle=h)
    assert h.check_device_error() == 0
    h.close()
    for c, r in enumerate(rows):
        assert torch.equal(B1[:r, c], B0[:r, c]), r
        assert torch.isinf(B1[r, c]), r
    assert torch.equal(B1[:, len(rows):], B0[:, len(rows):])
