"""FP64 TRSM leaves of 33 to 256 rows (few right-hand sides): orders at the edges of the
16-row blocks and of the leaf, right-hand sides at the edges of a CTA's 2, 4 and 8
columns and of the rule, both sides and directions; FP64 oracle. A row's Inf reaches no
row before it and no other column."""
import numpy as np
import pytest

from helpers import run_case, to_dev
from paper_2504_13821_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k", [33, 63, 65, 79, 80, 81, 127, 128, 129, 200, 255, 256, 257, 300])
@pytest.mark.parametrize("variant", ["LLNN", "LUNU", "LLTN", "RLNN", "RUTU"])
def test_edges(k, variant):
    side, uplo, trans, diag = variant
    for i, nrhs in enumerate((1, 2, 3, 303, 304, 305, 609, 1024, 1025)):
        m, n = (k, nrhs) if side == "L" else (nrhs, k)
        run_case("trsm", side, uplo, trans, diag, m, n, (1.0, -0.5)[i % 2], np.float64, k + nrhs,
                 lda_pad=i % 3, ldb_pad=i % 2)


@pytest.mark.parametrize("k", [100, 256])
def test_inf_stays_in_its_column_and_below(k):
    import paper_2504_13821_gb300 as trx
    A, B = inputs.problem("L", "L", k, 20, seed=k, dtype=np.float64)
    At, B0, B1 = (to_dev(z, "cuda:0") for z in (A, B, B))
    at = k - 40
    B1[at, 3] = float("inf")
    for z in (B0, B1):
        trx.trsm("L", "L", "N", "N", 1.0, At, z)
    rest = [c for c in range(20) if c != 3]
    assert torch.equal(B1[:at], B0[:at])
    assert torch.equal(B1[:, rest], B0[:, rest])
    assert not torch.isfinite(B1[at, 3])
