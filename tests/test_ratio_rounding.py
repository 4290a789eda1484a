"""CPU replay of the kernels' binary32 rounding of q / d (the Harris response):
the 32-bit digit division with a truncated reciprocal, the bits kept, the sticky
bit and the final scaling, against the oracle's correctly rounded ratio, on random values
of every magnitude, ties and near-ties, and every divisor the response takes."""
import numpy as np
import pytest

import oracle as O


def ratio(q, d):
    rcp = 0xFFFFFFFF // d
    if q == 0:
        return np.float32(0)
    m = abs(q)
    lz = 64 - m.bit_length()
    M = m << lz
    hi, lo = M >> 32, M & 0xFFFFFFFF
    q1 = (hi * rcp) >> 32
    r = hi - q1 * d
    assert 0 <= r < 2 * d
    if r >= d:
        q1, r = q1 + 1, r - d
    n = (r << 16) | (lo >> 16)
    assert n < 1 << 32
    q2 = (n * rcp) >> 32
    r = n - q2 * d
    assert 0 <= r < 2 * d and q2 < 1 << 16
    if r >= d:
        q2, r = q2 + 1, r - d
    nz = 32 - q1.bit_length()
    assert 0 <= nz <= 10
    rest = ((q2 << (16 + nz)) & 0xFFFFFFFF) | r | (lo & 0xFFFF)
    top = (q1 << nz) | (q2 >> (16 - nz)) | (1 if rest else 0)
    assert 1 << 31 <= top < 1 << 32
    # an integer to binary32, ties to even (numpy rounds integers once)
    f = np.float32(np.uint32(top)) * np.float32(2.0 ** (32 - lz - nz))
    return -f if q < 0 else f


@pytest.mark.parametrize("d", [1, 2, 3, 7, 16, 24, 25, 100, 255, 512, 999, 1000])
def test_ratio_to_float(d):
    rng = np.random.default_rng(d)
    qs = [int(rng.integers(1, 1 << int(b))) for b in rng.integers(2, 62, 1500)]
    for _ in range(500):  # at and next to the midpoints of neighbouring binary32 values
        M, e = int(rng.integers(1 << 23, 1 << 24)), int(rng.integers(0, 27))
        t = ((2 * M + 1) * d << e) >> 1
        qs += [t - 1, t, t + 1]
    qs = [q for q in qs + list(range(1, 300)) if 0 < q < 1 << 62]
    for q in qs:
        for s in (q, -q):
            assert ratio(s, d) == np.float32(O.round_ratio(s, d)), (s, d)


def test_every_divisor():
    rng = np.random.default_rng(1)
    for d in range(1, 1001):
        for b in (10, 34, 50, 61):
            q = int(rng.integers(1, 1 << b))
            assert ratio(q, d) == np.float32(O.round_ratio(q, d)), (q, d)
