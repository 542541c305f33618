"""FP32 side R on B's transpose in the workspace: at the edges of its 64x64
tiles and just above its smallest size, all side-R variants, padded ldb (the
padding untouched), against the oracle; and without the extra workspace, in
place, to the same bound."""
import numpy as np
import pytest

from helpers import run_case
from paper_2504_13821_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

RIGHT = [v for v in inputs.VARIANTS if v[0] == "R"]


@pytest.mark.parametrize("op", ["trsm", "trmm"])
@pytest.mark.parametrize("m,n", [(256, 256), (512, 512), (515, 511), (1025, 320), (2111, 257)])
def test_turned_against_oracle(op, m, n):
    import paper_2504_13821_gb300 as trx
    turned, plain = trx.Handle(0), trx.Handle(0)
    for h in (turned, plain):                    # the recursion at every size
        h.set_option(trx.OPT_THIN, -1)
        h.set_option(trx.OPT_THIN_LEAF, -1)
    need = turned.workspace_size("S" if op == "trsm" else "M", "R", m, n, 4)
    planes = turned.workspace_size("S" if op == "trsm" else "M", "L", n, m, 4)
    assert need > planes
    lib = trx.load_library()
    ws = torch.empty(planes, dtype=torch.uint8, device="cuda:0")
    for vi, v in enumerate(RIGHT):
        for h in (turned, plain):
            if h is plain:                       # the planes only: solved in place
                assert lib.trx_set_workspace(h.ptr, ws.data_ptr(), planes) == 0
                h._ws, h._ws_bytes = ws, 1 << 60
            run_case(op, *v, m, n, -1.5, np.float32, seed=inputs.variant_seed(n, vi), handle=h,
                     lda_pad=vi % 2, ldb_pad=(0, 3, 4)[vi % 3])
            assert h.check_device_error() == 0
    turned.close()
    plain.close()


@pytest.mark.parametrize("op", ["trsm", "trmm"])
def test_repeated_calls_on_other_arrays(op):
    """The cached launch graph belongs to one B: calls on another array, with
    another leading dimension, write that one."""
    import paper_2504_13821_gb300 as trx
    h = trx.Handle(0)
    h.set_option(trx.OPT_THIN, -1)
    h.set_option(trx.OPT_THIN_LEAF, -1)
    for seed, pad in ((1, 0), (2, 0), (3, 5), (1, 0)):
        for v in RIGHT[:4]:
            run_case(op, *v, 600, 500, 0.5, np.float32, seed=seed, handle=h, ldb_pad=pad)
    h.close()
