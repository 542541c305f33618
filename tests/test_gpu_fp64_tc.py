"""FP64 updates on the tensor cores (gemm_oz.cu) against DFMA and the oracle:
all variants at ragged sizes, one update alone element by element at tile,
chunk and K-step edges, rows that the fixed-point form cannot hold, and the
workspace rule.

Tolerances. An element the tensor cores compute is within 4 u sum |m||c| + u
|result| of the exact value, one left to DFMA within the bound of an FMA chain,
K u sum |m||c| + u |result| (u = 2^-53); sums in long double add less than u / 8.
"""
import numpy as np
import pytest

from helpers import run_case, to_dev
from paper_2504_13821_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

U = 2.0 ** -53


@pytest.fixture(scope="module")
def trx():
    import paper_2504_13821_gb300 as trx
    return trx


def one_update(trx, k1, m, n, side="L", edit=None, engine=0):
    """B2 + M B1 through TRMM with [[I, 0], [M, I]], I of order k1 rounded up to
    the recursion's split; returns (M, B1, B2, the lower rows of the result)."""
    k = k1 + m
    rng = np.random.default_rng(k + n)
    A = np.zeros((k, k), order="F")
    A[k1:, :k1] = rng.uniform(-1, 1, (m, k1)) / np.sqrt(k1)
    B = np.asfortranarray(rng.standard_normal((k, n)))
    if edit:
        edit(A[k1:, :k1], B[:k1])
    h = trx.Handle(0)
    h.set_option(trx.OPT_GEMM, engine)
    if side == "L":
        At, Bt = to_dev(A, "cuda:0"), to_dev(B, "cuda:0")
        trx.trmm("L", "L", "N", "U", 1.0, At, Bt, handle=h)
        out = Bt.cpu().numpy()
    else:                                   # B^T A^T: rows of C contiguous
        At, Bt = to_dev(A, "cuda:0"), to_dev(np.asfortranarray(B.T), "cuda:0")
        trx.trmm("R", "L", "T", "U", 1.0, At, Bt, handle=h)
        out = Bt.cpu().numpy().T
    assert h.check_device_error() == 0
    h.close()
    return A[k1:, :k1], B[:k1], B[k1:], out[k1:]


def errors(M, B1, B2, out, samples=400):
    """(error, sum |m||c|, |result|) of sampled elements, in long double."""
    rng = np.random.default_rng(5)
    i, j = rng.integers(0, M.shape[0], samples), rng.integers(0, B1.shape[1], samples)
    i[:4], j[:4] = [0, 0, -1, -1], [0, -1, 0, -1]
    p = M[i].astype(np.longdouble) * B1[:, j].T.astype(np.longdouble)
    exact = p.sum(1) + B2[i, j]
    return (np.abs(out[i, j] - exact).astype(float), np.abs(p).sum(1).astype(float),
            np.abs(exact).astype(float))


# (K, rows, right-hand sides): tile edges (128 rows; 64, 32 and 16 columns),
# exact chunks of 128 and ragged ones, every batch length of a last chunk
SIZES = [(256, 129, 640), (320, 200, 511), (384, 384, 1200), (448, 448, 97), (576, 300, 257),
         (640, 640, 33), (1024, 1000, 2049), (2048, 130, 300)]


@pytest.mark.parametrize("side", ["L", "R"])
@pytest.mark.parametrize("k1,m,n", SIZES)
def test_one_update_elementwise(trx, k1, m, n, side):
    err, mag, res = errors(*one_update(trx, k1, m, n, side))
    assert np.all(err <= 4.2 * U * mag + 1.1 * U * res)


@pytest.mark.parametrize("side", ["L", "R"])
def test_rows_of_wide_range(trx, side):
    """Columns graded over e^-40 against rows graded the other way: pieces the
    fixed-point form cannot hold are the FMA chain's."""
    k1, m, n = 512, 300, 400

    def edit(M, B1):
        g = np.exp(-40.0 * np.arange(k1) / k1)
        M[:, :] *= g[::-1]
        B1[:, 100:] *= g[:, None]
    err, mag, res = errors(*one_update(trx, k1, m, n, side, edit))
    assert np.all(err <= k1 * U * mag + 1.1 * U * res)


def test_extreme_and_special_values(trx):
    """Inf, NaN, zero rows and rows outside the exponent range: the same
    results as DFMA wherever that path computes them."""
    k1, m, n = 512, 300, 400

    def edit(M, B1):
        M[3, 5], M[40, 7], B1[9, 70] = np.inf, np.nan, -np.inf
        M[130, :] = 0.0
        M[200, :] *= 2.0 ** -400
        M[201, :] = 2.0 ** -1074
        B1[:, 300] *= 2.0 ** 700
        B1[:, 301] = 0.0
    M, B1, B2, out = one_update(trx, k1, m, n, "L", edit)
    ref = one_update(trx, k1, m, n, "L", edit, engine=1)[3]
    assert np.array_equal(np.isnan(out), np.isnan(ref))
    assert np.array_equal(np.isinf(out), np.isinf(ref))
    fine = np.isfinite(ref)
    with np.errstate(invalid="ignore", over="ignore"):
        mag = np.abs(np.where(np.isfinite(M), M, 0)) @ np.abs(np.where(np.isfinite(B1), B1, 0))
    assert np.all(np.abs(out - ref)[fine] <= ((2 * k1 * U) * mag + 4 * U * np.abs(ref))[fine])
    assert np.array_equal(out[130], ref[130], equal_nan=True)      # 0 * -Inf in column 70


@pytest.mark.parametrize("side,uplo,trans,diag", inputs.VARIANTS)
def test_all_variants(trx, side, uplo, trans, diag):
    h = trx.Handle(0)
    vi = inputs.VARIANTS.index((side, uplo, trans, diag))
    for op in ("trsm", "trmm"):
        k, nrhs = 701, 303
        m, n = (k, nrhs) if side == "L" else (nrhs, k)
        assert h.workspace_size("S" if op == "trsm" else "M", side, m, n, 8) > 0
        run_case(op, side, uplo, trans, diag, m, n, -1.5, np.float64,
                 seed=inputs.variant_seed(k, vi), handle=h, lda_pad=3, ldb_pad=1)
    assert h.check_device_error() == 0
    h.close()


def test_without_workspace_and_under_capture(trx):
    """No workspace: the DFMA result, bitwise; a stream capture on a fresh
    handle runs that way too; repeated calls agree bitwise."""
    k, n = 700, 300
    A, B = inputs.problem("L", "L", k, n, seed=9, dtype=np.float64)
    At, B0 = to_dev(A, "cuda:0"), to_dev(B, "cuda:0")
    dfma, fast, cap = trx.Handle(0), trx.Handle(0), trx.Handle(0)
    dfma.set_option(trx.OPT_GEMM, 1)
    assert dfma.workspace_size("S", "L", k, n, 8) == 0
    outs = {}
    for name, h in (("dfma", dfma), ("fast", fast), ("again", fast)):
        X = B0.clone()
        trx.trsm("L", "L", "N", "N", 1.5, At, X, handle=h)
        outs[name] = X.cpu().numpy()
    X = B0.clone()
    g = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(g):
        trx.trsm("L", "L", "N", "N", 1.5, At, X, handle=cap)
    g.replay()
    torch.cuda.synchronize()
    assert np.array_equal(X.cpu().numpy(), outs["dfma"])
    assert np.array_equal(outs["fast"], outs["again"])
    assert not np.array_equal(outs["fast"], outs["dfma"])
    for h in (dfma, fast, cap):
        h.close()


@pytest.mark.parametrize("side,uplo,trans,diag", inputs.VARIANTS)
def test_trmm_one_product(trx, side, uplo, trans, diag):
    """The whole FP64 TRMM at tile, step and chunk edges (128 rows, 16, 192),
    and across a scale segment (4096), against the oracle; repeatable."""
    h = trx.Handle(0)
    vi = inputs.VARIANTS.index((side, uplo, trans, diag))
    sizes = [(128, 1), (129, 70), (191, 16), (257, 200), (640, 33)]
    if vi in (0, 7, 10, 13):
        sizes.append((4200, 9))
    for k, nrhs in sizes:
        m, n = (k, nrhs) if side == "L" else (nrhs, k)
        out = [run_case("trmm", side, uplo, trans, diag, m, n, 1.5, np.float64,
                        seed=inputs.variant_seed(k, vi), handle=h, lda_pad=1, ldb_pad=vi % 3)[2]
               for _ in range(2)]
        assert np.array_equal(*out)
    assert h.check_device_error() == 0
    h.close()


def test_trmm_graded_columns(trx):
    """Right-hand sides that grow over e^60 down the column: pieces the
    fixed-point form cannot hold are computed from the kept original."""
    k, n = 700, 96
    A, B = inputs.problem("L", "L", k, n, seed=3, dtype=np.float64)
    A = np.asfortranarray(np.where(np.isnan(A), 0.0, A) * k)
    B = np.asfortranarray(B * np.exp(60.0 * np.arange(k) / k - 30.0)[:, None])
    At, Bt = to_dev(A, "cuda:0"), to_dev(B, "cuda:0")
    trx.trmm("L", "L", "N", "N", 1.0, At, Bt)
    L, out = np.tril(A).astype(np.longdouble), Bt.cpu().numpy()
    exact = L @ B.astype(np.longdouble)
    mag = np.abs(L) @ np.abs(B).astype(np.longdouble)
    assert np.all(np.abs(out - exact) <= k * U * mag)


@pytest.mark.parametrize("side,uplo,trans,diag", inputs.VARIANTS)
def test_refined_residual(trx, side, uplo, trans, diag):
    """FP32 TRSM with fixed corrections: the backward error of the result is at
    FP64 level (8 k u) with the tensor-core residual, and no larger than with the
    float-float one (CUDA cores)."""
    import oracle
    k, nrhs = 300, 70
    m, n = (k, nrhs) if side == "L" else (nrhs, k)
    vi = inputs.VARIANTS.index((side, uplo, trans, diag))
    A, B = inputs.problem(side, uplo, m, n, seed=inputs.variant_seed(k, vi), dtype=np.float32,
                          poison_diag=(diag == "U"))
    At, Bt = to_dev(A, "cuda:0"), to_dev(B, "cuda:0")
    eta = []
    for engine in (0, 1):
        h = trx.Handle(0)
        h.set_option(trx.OPT_GEMM, engine)
        X = trx.trsm_refined_async(side, uplo, trans, diag, 1.5, At, Bt, corrections=2, handle=h)
        torch.cuda.synchronize()
        assert h.check_device_error() == 0
        A64, B64 = np.asfortranarray(A.astype(np.float64)), np.asfortranarray(B.astype(np.float64))
        eta.append(oracle.trsm_backward_error(side, uplo, trans, diag, 1.5, A64,
                                              np.asfortranarray(X.cpu().numpy()), B64)["eta"])
        h.close()
    assert eta[0] <= 8 * k * U and eta[0] <= max(eta[1], 2 * U)
