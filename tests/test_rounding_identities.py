"""The FP32-pipe cuts of the packed kernel, in numpy binary32, against rounding on exact integers.

nearest-even: v k2 + rn(v k1) with k1 = 1 - 2^s, k2 = 2^s;  floor: v k2 + rz(v k1) with k1 = 1 + 2^s, k2 = -2^s (values of
at most 10 significant bits); s = 23 - M.  Both final additions are exact, so binary64 stands in for the FMA."""
import numpy as np
import pytest


def _mantissas():
    """24-bit significands: the ends of a binade, ties and near-ties of every M, and random ones."""
    rng = np.random.default_rng(5)
    edge = np.arange(1 << 13)
    m = [(1 << 23) + edge, (1 << 24) - 1 - edge, rng.integers(1 << 23, 1 << 24, 200000)]
    for bits in range(1, 11):
        tie = (1 << 23) + (rng.integers(0, 1 << bits, 2000) << (23 - bits)) + (1 << (22 - bits))
        m += [tie, tie - 1, tie + 1]
    return np.concatenate(m).astype(np.int64)


@pytest.mark.parametrize("M", range(1, 11))
def test_nearest_even_cut(M):
    m, s = _mantissas(), 23 - M
    v = (m / 2.0 ** 23).astype(np.float32)
    r = v * np.float32(1.0 - 2.0 ** s)
    got = v.astype(np.float64) * 2.0 ** s + r.astype(np.float64)
    q, rem, half = m >> s, m & ((1 << s) - 1), 1 << (s - 1)
    want = (q + ((rem > half) | ((rem == half) & (q & 1 == 1)))) * 2.0 ** -M
    assert (got == want).all()


@pytest.mark.parametrize("M", range(1, 9))
def test_floor_cut_of_short_products(M):
    m, s = np.arange(1 << 9, 1 << 10, dtype=np.int64), 23 - M
    exact = m * ((1 << s) + 1)                                   # v k1 in units of 2^-9
    sh = np.array([int(e).bit_length() - 24 for e in exact])
    r = (exact >> sh) << sh                                      # toward zero, 24 bits
    got = r - (m << s)
    assert (got == (m >> (9 - M)) << (9 - M)).all()
