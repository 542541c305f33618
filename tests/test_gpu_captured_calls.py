"""Calls captured into a caller's graph after the handle's buffers exist: replays are right
after larger calls on the handle have replaced them and their memory is in other hands.
The FP64 call depends on no workspace (it is the CUDA cores' result); the thin FP32 one
keeps its scratch."""
import numpy as np
import pytest

from helpers import to_dev
from paper_2504_13821_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def captured(handle, op, k, nrhs, dtype):
    """(replay, kept right-hand side, X) of one captured call."""
    import paper_2504_13821_gb300 as trx
    A, B = inputs.problem("L", "L", k, nrhs, seed=k, dtype=dtype)
    At, B0 = to_dev(A, "cuda:0"), to_dev(B, "cuda:0")
    X = B0.clone()
    run = lambda: getattr(trx, op)("L", "L", "N", "N", 1.5, At, X, handle=handle)
    run()                                            # the buffers exist
    first = X.clone()
    X.copy_(B0)
    g = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(g):
        run()
    return g, At, B0, X, first


def replay_after(handle, larger, g, B0, X):
    larger()                                         # replaces the handle's buffers
    torch.cuda.synchronize()
    junk = [torch.full((64 << 20,), 7, dtype=torch.uint8, device="cuda:0") for _ in range(8)]
    X.copy_(B0)
    g.replay()
    torch.cuda.synchronize()
    assert all(bool((j == 7).all()) for j in junk)
    assert handle.check_device_error() == 0
    return X.clone()


@pytest.mark.parametrize("op", ["trsm", "trmm"])
def test_f64(op):
    import paper_2504_13821_gb300 as trx
    h, dfma = trx.Handle(0), trx.Handle(0)
    dfma.set_option(trx.OPT_GEMM, 1)
    g, At, B0, X, first = captured(h, op, 700, 300, np.float64)
    big = to_dev(inputs.problem("L", "L", 2000, 900, seed=1, dtype=np.float64)[0], "cuda:0")
    Y = torch.ones((900, 2000), dtype=torch.float64, device="cuda:0").t()
    out = replay_after(h, lambda: getattr(trx, op)("L", "L", "N", "N", 1.0, big, Y, handle=h),
                       g, B0, X)
    ref = B0.clone()
    getattr(trx, op)("L", "L", "N", "N", 1.5, At, ref, handle=dfma)
    assert torch.equal(out, ref) and not torch.equal(first, ref)
    h.close()
    dfma.close()


@pytest.mark.parametrize("k,nrhs", [(512, 300), (2048, 600), (700, 16)])
def test_f32_thin(k, nrhs):
    import paper_2504_13821_gb300 as trx
    h = trx.Handle(0)
    g, At, B0, X, first = captured(h, "trsm", k, nrhs, np.float32)
    big = to_dev(inputs.problem("L", "L", 8192, 100, seed=1, dtype=np.float32)[0], "cuda:0")
    Y = torch.ones((100, 8192), dtype=torch.float32, device="cuda:0").t()
    ws = h._ws                                       # (FP32 planes: the caller's to keep)
    out = replay_after(h, lambda: trx.trsm("L", "L", "N", "N", 1.0, big, Y, handle=h), g, B0, X)
    assert torch.equal(out, first) and ws is not None
    h.close()
