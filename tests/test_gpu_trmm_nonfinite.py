"""TRMM with an Inf or NaN in the right-hand side: rows that do not depend on it are
those of the call without it, its own row and the rows below are Inf and NaN where the
CUDA cores' are. Positions inside and at the edges of the kernels' row tiles (4, 16, 32,
64, 128), orders of one and of several tiles, every tile width."""
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


@pytest.mark.parametrize("factor", [False, True], ids=["call", "factor"])
@pytest.mark.parametrize("variant", VARIANTS, ids="".join)
@pytest.mark.parametrize("k,n", [(256, 45), (300, 70), (700, 100), (1100, 45), (1100, 2200),
                                 (1100, 4400)])
def test_f32_by_rows(variant, k, n, factor):
    import paper_2504_13821_gb300 as trx
    m_, n_ = (k, n) if variant[0] == "L" else (n, k)
    A, B = inputs.problem(variant[0], variant[1], m_, n_, seed=k, dtype=np.float32,
                          poison_diag=variant[3] == "U")
    where = places(k)
    B1 = spoilt(B, *variant[:3], where)
    if factor:
        At, got = to_dev(A, "cuda:0"), []
        f = trx.Factor(*variant, At)
        for z in (B, B1):
            Bt = to_dev(z, "cuda:0")
            f.trmm(0.5, Bt)
            got.append(canonical(Bt.cpu().numpy(), *variant[:3]))
        f.close()
        clean, out = got
    else:
        clean, out = product(variant, A, B), product(variant, A, B1)
    ref = product(variant, A, B1, 1)
    assert np.array_equal(np.isnan(out), np.isnan(ref))
    assert np.array_equal(np.isposinf(out), np.isposinf(ref))
    assert np.array_equal(np.isneginf(out), np.isneginf(ref))
    for r, c, _ in where:
        assert np.array_equal(out[:r, c], clean[:r, c]) and not np.isfinite(out[r, c])
    rest = np.setdiff1d(np.arange(n), [c for _, c, _ in where])
    assert np.array_equal(out[:, rest], clean[:, rest])


@pytest.mark.parametrize("variant", VARIANTS[::3], ids="".join)
def test_f32_largest_finite_values(variant):
    """Entries that round to Inf in BF16 are no Inf: a row's sum has three roundings a term
    at most in the split form and k in the CUDA cores' chain, of |m||c| below 4e38 / k."""
    k, n = 400, 45
    m_, n_ = (k, n) if variant[0] == "L" else (n, k)
    A, B = inputs.problem(variant[0], variant[1], m_, n_, seed=4, dtype=np.float32)
    where = [(r, c, (-1) ** c * np.float32(3.4e38)) for c, r in enumerate(range(0, 400, 37))]
    B1 = spoilt(B, *variant[:3], where)
    out, ref = product(variant, A, B1), product(variant, A, B1, 1)
    fine = np.isfinite(ref)     # (not where diagonal times entry overflows before alpha)
    assert np.isfinite(out[fine]).all()
    assert np.abs(out.astype(float) - ref)[fine].max() <= 8 * k * 2.0 ** -24 * 3.4e38
