"""Batched problems (FP32, and FP64 cut over several CTAs) at the edges of the kernel's 16-row blocks, its 16-, 32- and
64-column chunks, the order where wide chunks end and the one where two blocks'
columns no longer fit together; right-hand sides cut over several CTAs; every
orientation; a batch larger than three rounds of the launch's CTAs (problems taken
ahead). Checked against the FP64 oracle with the 8 k u criteria."""
import itertools

import numpy as np
import pytest

from helpers import SENTINEL, bound, to_dev
import oracle
from paper_2504_13821_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

WAYS = list(itertools.product("SM", "LR", "LU", "NT", "NU"))


def run(shapes, seed, dtype=np.float32):
    import paper_2504_13821_gb300 as trx
    probs, host = [], []
    for i, (k, nrhs, (op, side, uplo, trans, diag), alpha) in enumerate(shapes):
        m, n = (k, nrhs) if side == "L" else (nrhs, k)
        A, B = inputs.problem(side, uplo, m, n, seed=seed + i, dtype=dtype,
                              poison_diag=(diag == "U"), lda=k + i % 4, ldb=m + i % 3)
        B[m:, :] = SENTINEL
        At, Bt = to_dev(A, "cuda:0"), to_dev(B, "cuda:0")
        probs.append((op, side, uplo, trans, diag, alpha, At[:k, :k], Bt[:m, :]))
        host.append((A, B, Bt))
    trx.batched(probs)
    torch.cuda.synchronize()
    for (k, nrhs, (op, side, uplo, trans, diag), alpha), (A, B, Bt) in zip(shapes, host):
        m = k if side == "L" else nrhs
        out = Bt.cpu().numpy()
        assert np.all(out[m:, :] == SENTINEL)
        X, Ak, B0 = (np.asfortranarray(z) for z in (out[:m], A[:k, :k], B[:m]))
        if op == "S":
            e = oracle.trsm_backward_error(side, uplo, trans, diag, alpha, Ak, X, B0)["eta"]
        else:
            ref = oracle.trmm(side, uplo, trans, diag, alpha, Ak, B0)
            e = oracle.trmm_error(side, uplo, trans, diag, alpha, Ak, X, ref, B0)
        assert np.isfinite(e) and e <= bound(k, dtype), (op, side, uplo, trans, diag, k, nrhs)


@pytest.mark.parametrize("k", [1, 2, 15, 16, 17, 33, 64, 127, 129, 255, 256, 257, 300, 395, 411,
                               511, 512])
def test_edges(k):
    widths = [1, 16, 17, 32, 33, 63, 64, 65, 150]
    shapes = [(k, widths[(i + k) % len(widths)], way, (1.0, -0.5)[i % 2])
              for i, way in enumerate(WAYS)]
    run(shapes, 1000 * k)


@pytest.mark.parametrize("k", [1, 17, 130, 512])
def test_f64_cut_over_ctas(k):
    widths = [1, 15, 16, 17, 64, 77, 300]
    shapes = [(k, widths[i % 7], way, (1.0, -0.5)[i % 2]) for i, way in enumerate(WAYS)]
    shapes.append((40, 9000, WAYS[k % 32], 1.0))
    run(shapes, 1000 * k, np.float64)


def test_many_problems_and_wide_right_hand_sides():
    rng = np.random.default_rng(3)
    shapes = [(int(rng.integers(1, 40)), int(rng.integers(1, 40)), WAYS[int(rng.integers(32))], 1.0)
              for _ in range(1800)]
    shapes += [(40, 20000, WAYS[0], 2.0), (300, 2000, WAYS[21], 1.0)]
    run(shapes, 7)


@pytest.mark.parametrize("k", [16, 40, 256, 300, 512])
@pytest.mark.parametrize("op", ["S", "M"])
def test_infinite_rows_reach_only_the_rows_that_use_them(op, k):
    """Lower, not transposed: row i of the result depends on rows <= i only."""
    import paper_2504_13821_gb300 as trx
    A, B = inputs.problem("L", "L", k, 40, seed=k, dtype=np.float32)
    at = k - 3
    At, B0, B1 = (to_dev(z, "cuda:0") for z in (A, B, B))
    B1[at, 5] = float("inf")
    trx.batched([(op, "L", "L", "N", "N", 1.0, At, z) for z in (B0, B1)])
    assert torch.equal(B1[:at], B0[:at])
    rest = [c for c in range(40) if c != 5]
    assert torch.equal(B1[:, rest], B0[:, rest])
    assert not torch.isfinite(B1[at:, 5]).any()
