"""The thin TRSM's bounded waits run out together: with block row 0 never published,
every later block row's wait ends, all the threads of a CTA leave at the same step, the
launch reports TRX_ERR_TIMEOUT, and the next call is right. Repeated over chain lengths
and panel counts, as which thread sees the stop first differs from run to run."""
import numpy as np
import pytest

from helpers import run_case

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k,nrhs", [(128, 16), (577, 50), (2048, 64), (4096, 200), (8191, 16)])
def test_timeouts_end(k, nrhs):
    import paper_2504_13821_gb300 as trx
    from paper_2504_13821_gb300 import _binding
    h = trx.Handle(0)
    h.set_option(trx.OPT_THIN, 1)
    h.set_option(trx.OPT_GRAPH, 0)
    for limit in (1000, 20_000, 300_000):                 # ns
        h.set_option(trx.OPT_WAIT_LIMIT, limit)
        h.set_option(_binding.OPT_TEST_WITHHOLD, 1)
        for _ in range(5):
            run_case("trsm", "L", "L", "N", "N", k, nrhs, 1.0, np.float32, seed=k, handle=h,
                     check=False)
            assert h.check_device_error() == 4            # TRX_ERR_TIMEOUT
    h.set_option(_binding.OPT_TEST_WITHHOLD, 0)
    h.set_option(trx.OPT_WAIT_LIMIT, 2_000_000_000)
    run_case("trsm", "L", "L", "N", "N", k, nrhs, 1.0, np.float32, seed=k, handle=h)
    assert h.check_device_error() == 0
    h.close()
