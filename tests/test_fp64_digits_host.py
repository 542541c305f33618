"""The arithmetic of the FP64 tensor-core update (gemm_oz.cu) replayed on the
host: the digits of a scaled row, the level sums of a K chunk, their carries in
FP32 and the running sums, against exact rational arithmetic."""
from fractions import Fraction

import numpy as np
import pytest


def digits(row):
    """(e, digits[l][8]) of a row: x = 2^e sum_s d_s 2^-8s, rounded to 64 bits."""
    e = int(np.frexp(np.abs(row).max())[1]) + 1          # |x| 2^-e < 1/2
    out = []
    for x in row:
        q = Fraction(float(x)) * Fraction(2) ** (64 - e)
        q = int(abs(q) + Fraction(1, 2)) * (1 if q >= 0 else -1)
        low = (q & ((1 << 56) - 1)) + 0x80808080808080
        d = [(q >> 56) + (low >> 56)]
        d += [((low >> (8 * b)) & 255) - 128 for b in range(6, -1, -1)]
        assert sum(v << (56 - 8 * s) for s, v in enumerate(d)) == q
        assert max(map(abs, d)) <= 128
        out.append(d)
    return e, np.array(out, dtype=np.int64)


def update(a, b):
    """sum a b as the kernel forms it: chunks of 192, levels 2..9, FP32 carries."""
    f32, magic = np.float32, np.float32(12582912.0)
    (ea, da), (eb, db) = digits(a), digits(b)
    T, R = 0, f32(0)
    for k0 in range(0, len(a), 192):
        lev = {s: 0 for s in range(2, 10)}
        for i in range(1, 9):
            for j in range(1, 10 - i):
                lev[i + j] += int((da[k0:k0 + 192, i - 1] * db[k0:k0 + 192, j - 1]).sum())
        # exact in FP32; the lowest three, where they pass 2^24, to their last bits
        assert all(abs(lev[s]) <= 1 << 24 for s in range(2, 7)) and abs(lev[2]) <= 1 << 22
        lev.update({s: int(f32(lev[s])) for s in (7, 8, 9)})
        T += (lev[5] << 8) + (lev[4] << 16) + (lev[3] << 24) + (lev[2] << 32)
        g8 = f32(float(lev[9]) * 2.0 ** -8 + lev[8])
        t8 = f32(float(g8) * 2.0 ** -8 + float(magic)) - magic
        g7 = f32(lev[7]) + t8
        t7 = f32(float(g7) * 2.0 ** -8 + float(magic)) - magic
        R = f32(R + f32(float(t8) * -256.0 + float(g8)))
        R = f32(float(f32(float(t7) * -256.0 + float(g7))) * 256.0 + float(R))
        assert abs(float(R)) <= 2.0 ** 24
        T += int(round(float(f32(lev[6]) + t7)))
        assert abs(T) < 1 << 63
    return (Fraction(T) / 2 ** 48 + Fraction(int(round(float(R)))) / 2 ** 64) * \
        Fraction(2) ** (ea + eb), ea + eb


def rows(kind, K, rng):
    if kind == "normal":
        return rng.standard_normal(K), rng.uniform(-1, 1, K)
    if kind == "largest digits":             # every digit product near its bound
        x = float((sum(128 * 2.0 ** (-8 * s) for s in range(1, 8)) - 2.0 ** -8) *
                  (1 - 2.0 ** -53))
        return np.full(K, x), np.full(K, -x)
    if kind == "top digit carries":          # mantissas just below a power of two
        return np.nextafter(np.ones(K), 0), -np.nextafter(np.ones(K) * 4, 0)
    return np.exp(rng.uniform(-40, 0, K)) * rng.choice([-1, 1], K), rng.standard_normal(K)


@pytest.mark.parametrize("kind", ["normal", "largest digits", "top digit carries", "wide"])
@pytest.mark.parametrize("K", [1, 191, 192, 193, 700])
def test_update_error(kind, K):
    """|error| <= K 2^-62 in units of the scaled operands."""
    a, b = rows(kind, K, np.random.default_rng(K))
    got, e = update(a, b)
    exact = sum(Fraction(float(x)) * Fraction(float(y)) for x, y in zip(a, b))
    assert abs(got - exact) <= K * Fraction(2) ** (e - 62)
