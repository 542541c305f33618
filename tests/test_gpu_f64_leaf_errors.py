"""The two FP64 TRSM leaf kernels (up to and from 1024 right-hand sides on) solve the same
columns with errors of the same size, against long double. Both sum a block's 16
products before they meet a row, so a row takes as many roundings of its own size in
one as in the other: their errors differ by the order inside those sums only, below a
quarter of each other over thousands of elements (16 roundings at the row's size
would be 1.6 times the error)."""
import numpy as np
import pytest

from helpers import to_dev

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k", [64, 512])
def test_errors_of_both_leaves(k):
    import paper_2504_13821_gb300 as trx
    rng = np.random.default_rng(k)
    A = np.tril(rng.uniform(-1, 1, (k, k)), -1) / np.sqrt(k)
    A += np.diag(1 + np.abs(rng.standard_normal(k)))
    B = rng.standard_normal((k, 2048))
    h = trx.Handle(0)
    h.set_option(trx.OPT_LEAF, 64)
    h.set_option(trx.OPT_GEMM, 1)
    cols = 64
    L, X = A.astype(np.longdouble), np.empty((k, cols), np.longdouble)
    for i in range(k):
        X[i] = (B[i, :cols] - L[i, :i] @ X[:i]) / L[i, i]
    err = []
    for n in (1024, 2048):
        At, Bt = (to_dev(np.asfortranarray(z), "cuda:0") for z in (A, B[:, :n]))
        trx.trsm("L", "L", "N", "N", 1.0, At, Bt, handle=h)
        d = Bt[:, :cols].cpu().numpy() - X
        err.append(float(np.sqrt((d * d).sum() / (X * X).sum())))
    h.close()
    assert err[1] <= 1.25 * err[0], err
