"""The automatic thin solve and thin leaves around their lines (order 256 and 1024,
1024 and 1536 right-hand sides, twice the order, 2^20 elements): both sides, forward and
reversed, plain calls, a prepared factor and capture of a call that has not run before,
against the FP64 oracle; an explicit option keeps the recursion."""
import numpy as np
import pytest

from helpers import run_case, to_dev
from paper_2504_13821_gb300 import debug_plan, inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k,nrhs", [(255, 300), (256, 512), (256, 513), (257, 514), (300, 601),
                                    (682, 1536), (683, 1536), (1023, 1200), (1024, 1024),
                                    (1025, 1024), (1024, 1025), (1030, 1537), (2049, 257),
                                    (2100, 700)])
@pytest.mark.parametrize("variant", ["LLNN", "LUNU", "RLNN", "RUTN"])
def test_lines(k, nrhs, variant):
    side, uplo, trans, diag = variant
    m, n = (k, nrhs) if side == "L" else (nrhs, k)
    run_case("trsm", side, uplo, trans, diag, m, n, -0.5, np.float32, k + nrhs, lda_pad=1, ldb_pad=3)


@pytest.mark.parametrize("k,nrhs", [(300, 600), (1536, 800)])
def test_factor_and_first_call_in_a_capture(k, nrhs):
    import paper_2504_13821_gb300 as trx
    A, B = inputs.problem("L", "L", k, nrhs, seed=k, dtype=np.float32)
    At, X, Y, Z = (to_dev(z, "cuda:0") for z in (A, B, B, B))
    trx.trsm("L", "L", "N", "N", 1.0, At, X)
    f = trx.Factor("L", "L", "N", "N", At)
    f.trsm(1.0, Y)
    assert torch.equal(X, Y)
    # no scratch yet: the capture holds the recursion, which the thin solve agrees with
    h = trx.Handle(0)
    h.ensure_workspace(h.workspace_size("S", "L", k, nrhs, 4))
    s, g = torch.cuda.Stream(), torch.cuda.CUDAGraph()
    s.wait_stream(torch.cuda.current_stream())
    with torch.cuda.graph(g, stream=s):
        trx.trsm("L", "L", "N", "N", 1.0, At, Z, handle=h)
    Z.copy_(to_dev(B, "cuda:0"))
    g.replay()
    torch.cuda.synchronize()
    assert (Z - X).abs().max() <= 16 * k * 2.0 ** -24 * X.abs().max()


def test_explicit_leaf_keeps_the_recursion():
    for leaf, kinds in ((0, {"thin"}), (128, {"leaf"})):
        steps = debug_plan("S", "L", "L", "N", "N", 2048, 700, 4, leaf, 0)
        assert {s["kind"] for s in steps} & {"thin", "leaf"} == kinds
