"""FP64 updates on the tensor cores where their error bound is nearest: rows and columns with
one large entry each in different places and small ones of adverse digits, just above
the line where the product is left to DFMA. An element's error is below 8 u sum |m||c| +
u |result|, u = 2^-53: K' 2^-62 in units of the scaled operands, at sums of at least K'
2^-12. On the host replay of the same rows it is above 2 u, so the line is near."""
from fractions import Fraction

import numpy as np
import pytest

from test_fp64_digits_host import digits, update

U = 2.0 ** -53


def adverse(K, top, low, last):
    x = float(sum(Fraction(d, 256 ** (s + 1)) for s, d in enumerate([top] + 6 * [low] + [last])))
    a, b = np.full(K, x), np.full(K, x)
    a[0] = b[1] = 0.499999
    return a, b


def magnitudes(a):
    """As the kernel's: BF16 rounded down, over the row's power of two."""
    m, e = np.frexp(np.abs(a))
    return np.ldexp(np.floor(m * 256) / 256, e - digits(a)[0])


@pytest.mark.parametrize("K,top,last", [(256, 4, 96), (704, 4, 96)])
def test_host_replay(K, top, last):
    a, b = adverse(K, top, 127, last)
    assert 1 <= (magnitudes(a) @ magnitudes(b)) / (K * 2.0 ** -12) < 1.6
    got, _ = update(a, b)
    terms = [Fraction(float(x)) * Fraction(float(y)) for x, y in zip(a, b)]
    err = abs(got - sum(terms)) / sum(map(abs, terms))
    assert 2 * U < err <= 8 * U


@pytest.mark.gpu
@pytest.mark.parametrize("K,top,last", [(256, 4, 96), (704, 4, 96)])
def test_one_update(K, top, last):
    import paper_2504_13821_gb300 as trx
    from test_gpu_fp64_tc import errors, one_update
    a, b = adverse(K, top, 127, last)

    def edit(M, B1):
        rng = np.random.default_rng(K)
        M[:], B1[:] = a, 1024 * b[:, None]          # (B2's entries stay small beside B1's)
        M[::3] *= -1
        M[:, 2:] = M[:, 2:][:, rng.permutation(K - 2)]
    args = (trx, K, 130, 300, "L", edit)
    M, B1, B2, out = one_update(*args)
    assert not np.array_equal(out, one_update(*args, engine=1)[3])
    err, mag, res = errors(M, B1, B2, out)
    assert np.all(err <= 8 * U * mag + 1.1 * U * res)
