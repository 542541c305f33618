"""Few right-hand sides in FP32 with ill-conditioned diagonal blocks: the thin solve's
backward error is that of the recursion, which substitutes. Diagonal blocks of 64 rows
with entries up to 1 below a diagonal 1 + |N(0,1)| (inverted and multiplied, such a
block leaves about 8 times substitution's error), small entries elsewhere, right-hand
sides M x of a known x. Both errors are the largest of thousands of elements' and a few
u each, so they differ by less than a factor of 2.5 when both substitute."""
import numpy as np
import pytest

from helpers import to_dev

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def triangle(k, rng):
    """Lower triangle with ill-conditioned 64-row blocks on the diagonal."""
    A = np.tril(rng.uniform(-1, 1, (k, k)), -1) / k
    for i in range(0, k, 64):
        b = A[i:i + 64, i:i + 64]
        b *= k
        b += np.diag(1 + np.abs(rng.standard_normal(len(b))))
    return A.astype(np.float32)


@pytest.mark.parametrize("k,nrhs,upper", [(256, 100, False), (512, 300, True), (577, 16, False),
                                          (1000, 400, False), (1024, 64, True),
                                          (2048, 600, False)])
def test_backward_error_of_the_recursion(k, nrhs, upper):
    import paper_2504_13821_gb300 as trx
    rng = np.random.default_rng(k)
    L = triangle(k, rng)
    x = rng.standard_normal((k, nrhs)).astype(np.float32)
    B = (L.astype(float) @ x).astype(np.float32)
    if upper:                                   # the same problem, its rows reversed
        L, B = np.ascontiguousarray(L[::-1, ::-1]), np.ascontiguousarray(B[::-1])
    err = []
    for off in (0, -1):
        h = trx.Handle(0)
        h.set_option(trx.OPT_THIN, off)
        h.set_option(trx.OPT_THIN_LEAF, off)
        At, Bt = to_dev(np.asfortranarray(L), "cuda:0"), to_dev(np.asfortranarray(B), "cuda:0")
        trx.trsm("L", "U" if upper else "L", "N", "N", 1.0, At, Bt, handle=h)
        assert h.check_device_error() == 0
        h.close()
        X = Bt.cpu().numpy().astype(float)
        A64 = L.astype(float)
        err.append((np.abs(B - A64 @ X) / (np.abs(A64) @ np.abs(X))).max())
    assert err[0] <= 2.5 * err[1], err
