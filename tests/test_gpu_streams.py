"""Calls of several handles on several streams at once, each repeated, give bitwise
the results of the same calls one after the other. Sizes at which the update
kernels' tiles are narrower than 256 columns and few enough that the streams' launches
share the SMs, with and without column-panel branches inside a call."""
import numpy as np
import pytest

from helpers import to_dev
from paper_2504_13821_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# (operation, side, uplo, trans, order, right-hand sides, column panels)
F32 = [("trsm", "L", "L", "N", 1000, 3000, 0), ("trsm", "L", "L", "N", 1000, 3000, 3),
       ("trmm", "R", "U", "T", 700, 900, 0), ("trsm", "R", "L", "N", 2048, 1700, 0)]
F64 = [("trsm", "L", "L", "N", 1000, 200, 0), ("trsm", "R", "U", "N", 1024, 1500, 0),
       ("trmm", "L", "U", "T", 700, 300, 0), ("trmm", "R", "L", "N", 300, 40, 0)]


def together(calls, dtype, rounds=6):
    import paper_2504_13821_gb300 as trx
    jobs = []
    for i, (op, side, uplo, trans, k, nrhs, panels) in enumerate(calls):
        m, n = (k, nrhs) if side == "L" else (nrhs, k)
        A, B = inputs.problem(side, uplo, m, n, seed=100 + i, dtype=dtype)
        h = trx.Handle(0)
        if panels:
            h.set_option(trx.OPT_PANELS, panels)
        At, B0 = to_dev(A, "cuda:0"), to_dev(B, "cuda:0")
        alone, out = B0.clone(), B0.clone()
        run = lambda X, s, op=op, side=side, uplo=uplo, trans=trans, At=At, h=h: getattr(trx, op)(
            side, uplo, trans, "N", 1.5, At, X, handle=h, stream=s)
        run(alone, torch.cuda.current_stream())
        torch.cuda.synchronize()
        assert torch.isfinite(alone).all()
        jobs.append((run, B0, alone, out, torch.cuda.Stream(), h))
    for _ in range(rounds):
        for run, B0, _, out, s, _ in jobs:
            with torch.cuda.stream(s):
                out.copy_(B0)
            run(out, s)
        torch.cuda.synchronize()
        for _, _, alone, out, _, h in jobs:
            assert h.check_device_error() == 0
            assert torch.equal(out, alone)
    for job in jobs:
        job[-1].close()


def test_f32_calls_on_several_streams():
    together(F32, np.float32)


def test_f64_calls_on_several_streams():
    together(F64, np.float64)


def test_f32_and_f64_calls_at_once():
    import threading
    failed = []

    def work(calls, dtype):
        try:
            together(calls, dtype, rounds=3)
        except BaseException as e:
            failed.append(e)
    threads = [threading.Thread(target=work, args=a) for a in ((F32[:2], np.float32),
                                                               (F64[:2], np.float64))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed, failed
