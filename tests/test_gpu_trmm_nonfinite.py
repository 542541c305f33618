"""TRMM with an Inf or NaN in the right-hand side: rows that do not depend on it are
those of the call without it, its own row and the rows below are the CUDA cores'
results (FP64) or not finite where those are not (FP32). Positions inside and at the edges of
the kernels' row tiles (4, 16, 32, 64, 128), orders of one and of several tiles."""
import numpy as np
import pytest

from helpers import to_dev
from paper_2504_13821_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

VARIANTS = [("L", "L", "N", "N"), ("L", "U", "N", "U"), ("L", "L", "T", "N"),
            ("R", "L", "N", "N"), ("R", "U", "T", "U")]


def canonical(X, side, uplo, trans):
    """The result as the canonical lower problem has it: order by right-hand sides, a
    row depending on the rows before it."""
    Y = X if side == "L" else X.T
    forward = (uplo == "L") == ((trans == "N") == (side == "L"))
    return Y if forward else Y[::-1]


def spoilt(B, side, uplo, trans, places):
    B = B.copy(order="F")
    V = canonical(B, side, uplo, trans)
    for r, c, v in places:
        V[r, c] = v
    return B


def product(variant, A, B, engine=0):
    import paper_2504_13821_gb300 as trx
    h = trx.Handle(0)
    h.set_option(trx.OPT_GEMM, engine)
    At, Bt = to_dev(A, "cuda:0"), to_dev(B, "cuda:0")
    trx.trmm(*variant, 0.5, At, Bt, handle=h)
    assert h.check_device_error() == 0
    h.close()
    return canonical(Bt.cpu().numpy(), *variant[:3])


def places(k):
    at = [0, 1, 18, 63, 64, 77, 127, 131, k // 2 + 5, k - 2]
    return [(min(r, k - 1), 3 * i + 1, (np.inf, np.nan, -np.inf)[i % 3])
            for i, r in enumerate(at)]


@pytest.mark.parametrize("variant", VARIANTS, ids="".join)
@pytest.mark.parametrize("k", [128, 200, 300, 700])
def test_f64(variant, k):
    n = 45
    m_, n_ = (k, n) if variant[0] == "L" else (n, k)
    A, B = inputs.problem(variant[0], variant[1], m_, n_, seed=k, dtype=np.float64,
                          poison_diag=variant[3] == "U")
    where = places(k)
    B1 = spoilt(B, *variant[:3], where)
    clean, out, ref = (product(variant, A, z, e) for z, e in ((B, 0), (B1, 0), (B1, 1)))
    assert np.array_equal(np.isnan(out), np.isnan(ref))
    assert np.array_equal(np.isposinf(out), np.isposinf(ref))
    assert np.array_equal(np.isneginf(out), np.isneginf(ref))
    fine = np.isfinite(ref)
    # two FMA chains, or one and a product of digits: k u sum |m||c| each, and a row's sum
    # is at most (max|diagonal| + 1) max|c| (off-diagonal entries below 1 / k)
    tol = 4 * k * 2.0 ** -53 * np.abs(B).max() * (np.nanmax(np.abs(A)) + 1)
    for r, c, _ in where:
        assert np.all(fine[:r, c]) and not fine[r, c]
        assert np.abs(out[:r, c] - clean[:r, c]).max(initial=0.0) <= tol
    assert np.abs(out - ref)[fine].max() <= tol
