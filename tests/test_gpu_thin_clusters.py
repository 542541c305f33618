"""FP32 TRSM with few right-hand sides: orders around the 64-row blocks and the eight
block rows of a cluster, with M's columns aligned (16-byte copies) and not, both
contiguous directions, one panel and several; against the FP64 oracle. An Inf in the
right-hand side stays in its own column and out of the block rows before it."""
import numpy as np
import pytest

from helpers import run_case, to_dev
from paper_2504_13821_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def handle():
    import paper_2504_13821_gb300 as trx
    h = trx.Handle(0)
    h.set_option(trx.OPT_THIN, 1)
    yield h
    h.close()


@pytest.mark.parametrize("k", [63, 64, 65, 128, 130, 447, 511, 512, 513, 577, 1024, 1087])
@pytest.mark.parametrize("variant", ["LLNN", "LUNU", "LLTN", "LUTN", "RLNN", "RUTU"])
def test_edges(handle, k, variant):
    side, uplo, trans, diag = variant
    for i, nrhs in enumerate((1, 16, 17, 50)):
        m, n = (k, nrhs) if side == "L" else (nrhs, k)
        run_case("trsm", side, uplo, trans, diag, m, n, (1.0, -0.5)[i % 2], np.float32, k + nrhs,
                 lda_pad=(-k) % 4 if i % 2 else 1, ldb_pad=i, handle=handle)


@pytest.mark.parametrize("op", ["trsm", "trmm"])
def test_inf_stays_in_its_column_and_below(handle, op):
    import paper_2504_13821_gb300 as trx
    k, at = 900, 700
    A, B = inputs.problem("L", "L", k, 20, seed=5, dtype=np.float32)
    At, B0, B1 = (to_dev(z, "cuda:0") for z in (A, B, B))
    B1[at, 3] = float("inf")
    for z in (B0, B1):
        getattr(trx, op)("L", "L", "N", "N", 1.0, At, z, handle=handle)
    rest = [c for c in range(20) if c != 3]
    first = at // 4 * 4                    # the products take four rows at a time
    assert torch.equal(B1[:first], B0[:first])
    assert torch.equal(B1[:, rest], B0[:, rest])
    assert not torch.isfinite(B1[at, 3])
