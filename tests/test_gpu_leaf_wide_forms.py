"""The 128-row leaf for many right-hand sides in the forms its staging and write-back
tell apart: both contiguous directions of A, rows of B forwards, reversed and strided,
columns that start on 16 bytes and that do not, ragged last blocks; FP64 oracle."""
import numpy as np
import pytest

from helpers import run_case

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k", [260, 384, 397])
@pytest.mark.parametrize("variant", ["LLNN", "LUNU", "LLTN", "LUTU", "RLNN", "RUTN"])
@pytest.mark.parametrize("pad", [0, 1, 4])
def test_forms(k, variant, pad):
    side, uplo, trans, diag = variant
    m, n = (k, 1603) if side == "L" else (1603, k)
    run_case("trsm", side, uplo, trans, diag, m, n, -1.5, np.float32, k + pad, lda_pad=pad, ldb_pad=pad)
