"""The division-free forms of m / 6 that the kernels use, against the division.

fl(m/6) by one residual step, and floor_E4M3(fl(m/6)) from the product with
fl(1/6) rounded towards zero, over every mantissa of two octaves (both are
scale-free in the normal range) and every fp32 from below the smallest E4M3 code
to above the largest, in steps that visit every rounding boundary.
"""
import numpy as np

SIXTH = np.array([0x3E2AAAAB], dtype=np.uint32).view(np.float32)[0]


def floor_code(s):
    """Largest E4M3 code whose value is at most s."""
    v = np.array([c * 2.0 ** -9 if c < 8 else (1 + (c & 7) / 8) * 2.0 ** ((c >> 3) - 7) for c in range(127)])
    return np.searchsorted(v, s.astype(np.float64), side="right") - 1


def mul_rz(a):
    p = a.astype(np.float64) * np.float64(SIXTH)             # exact: 48 bits
    f = p.astype(np.float32)
    b = f.view(np.uint32).copy()
    b[f.astype(np.float64) > p] -= 1
    return b.view(np.float32)


def floor_code_of_sixth(m):
    s = mul_rz(m)
    sub = np.floor(s.astype(np.float64) * 512).astype(np.int64) & 0xFF
    top = (s.view(np.uint32) >> 20).astype(np.int64) - 960
    return np.minimum(np.where(s < np.float32(0.03125), sub, top), 126)


def sixth(m):
    q = m * SIXTH
    rem = (m.astype(np.float64) - 6.0 * q.astype(np.float64)).astype(np.float32)
    return (rem.astype(np.float64) * np.float64(SIXTH) + q.astype(np.float64)).astype(np.float32)


def around(values):
    """fp32 neighbours of 6 v, four on each side."""
    b = (6.0 * values).astype(np.float32).view(np.uint32).astype(np.int64)
    return (b[:, None] + np.arange(-4, 5)[None, :]).reshape(-1).astype(np.uint32).view(np.float32)


def test_every_mantissa():
    for e in (124, 127):
        m = (np.arange(1 << 23, dtype=np.uint32) | np.uint32(e << 23)).view(np.float32)
        assert np.array_equal(sixth(m), m / np.float32(6))
        assert np.array_equal(floor_code_of_sixth(m), floor_code(m / np.float32(6)))


def test_every_code_boundary():
    codes = np.array([c * 2.0 ** -9 if c < 8 else (1 + (c & 7) / 8) * 2.0 ** ((c >> 3) - 7) for c in range(1, 127)])
    mids = (codes[1:] + codes[:-1]) / 2
    m = np.concatenate([around(codes), around(mids), np.float32([0.0, 1e-30, 5e3, 1e9, 2.0 ** 47])])
    assert np.array_equal(floor_code_of_sixth(m), np.minimum(floor_code(m / np.float32(6)), 126))
    big = m[m > 1e-20]
    assert np.array_equal(sixth(big), big / np.float32(6))


def test_planted_rounding_is_caught():
    """Rounding the product to nearest instead of towards zero moves a code."""
    m = around(np.array([1.25]))
    s = m * SIXTH
    wrong = np.minimum((s.view(np.uint32) >> 20).astype(np.int64) - 960, 126)
    assert not np.array_equal(wrong, floor_code(m / np.float32(6)))
