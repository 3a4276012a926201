"""The division by a constant of the path decoding: for every divisor the kernels meet (tiles per row, items
of a wave segment), q = (n * mul) >> 32 >> (shift - 1) equals n // d for 0 <= n < 2^31."""
import numpy as np
import pytest


def make(d):
    if d <= 1:
        return 0, -1
    l = 0
    while (1 << l) < d:
        l += 1
    mul = ((1 << (31 + l)) // d) + 1
    assert mul < 1 << 32
    return mul, l


@pytest.mark.parametrize("d", [1, 2, 3, 5, 7, 8, 26, 31, 32, 33, 240, 480, 641, 65535, 65536, 131072, 524288, 518144,
                               (1 << 26) - 1, 1 << 26, (1 << 30) + 1, (1 << 31) - 1])
def test_fast_div(d):
    mul, shift = make(d)
    rng = np.random.default_rng(d)
    n = np.concatenate([rng.integers(0, 1 << 31, 20000), np.arange(200), [(1 << 31) - 1]])
    k = rng.integers(0, (1 << 31) // d, 20000) * d
    n = np.unique(np.clip(np.concatenate([n, k, k - 1, k + d - 1]), 0, (1 << 31) - 1)).astype(np.uint64)
    q = n if shift < 0 else ((n * np.uint64(mul)) >> np.uint64(32)) >> np.uint64(shift - 1)
    assert np.array_equal(q, n // np.uint64(d))
