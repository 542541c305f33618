"""The one-launch TRMM (the recursion's updates gathered by 128-row tile) at the
edges of its tiles, K steps and 256-term chunks and of its scheduling rounds,
against the oracle (8 k u) and bitwise repeatable."""
import numpy as np
import pytest

from helpers import run_case
from paper_2504_13821_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# orders around 128-row tiles and 256-term chunks; right-hand sides from just
# above the thin product's range to several rounds of tiles per CTA
SIZES = [(256, 33), (257, 64), (383, 65), (385, 129), (511, 1000), (513, 257), (1023, 2100),
         (1281, 520), (2049, 1500)]


@pytest.mark.parametrize("k,nrhs", SIZES)
def test_sizes_against_oracle(k, nrhs):
    import paper_2504_13821_gb300 as trx
    variants = inputs.VARIANTS if k < 600 else inputs.VARIANTS[::5]
    h = trx.Handle(0)
    for vi, v in enumerate(variants):
        m, n = (k, nrhs) if v[0] == "L" else (nrhs, k)
        seed = inputs.variant_seed(k, vi)
        _, _, X = run_case("trmm", *v, m, n, 1.5, np.float32, seed=seed, handle=h, ldb_pad=vi % 3)
        _, _, Y = run_case("trmm", *v, m, n, 1.5, np.float32, seed=seed, handle=h, ldb_pad=vi % 3,
                           check=False)
        assert np.array_equal(X, Y)
    h.close()
