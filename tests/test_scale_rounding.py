"""The division-free forms of m / 6 that the kernels use, against the division.

In numpy: fl(m/6) by one residual step over every mantissa of two octaves (it is
scale-free in the normal range), and floor_E4M3(fl(m/6)) from the product with
fl(1/6) rounded towards zero over every fp32 from the octave of six times the
smallest E4M3 code to that of six times the largest.  On a GPU: the kernels' own
forms, through blocks whose largest element is a neighbour of a code's or a
midpoint's sixfold, or any fp32 between.
"""
import numpy as np
import pytest
import torch

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
    for e in range(120, 139):                               # 2^-7 <= m < 2^12: 6 v from 1.5 2^-7 to 1.3125 2^11
        m = (np.arange(1 << 23, dtype=np.uint32) | np.uint32(e << 23)).view(np.float32)
        s = m / np.float32(6)
        if e in (124, 127):
            assert np.array_equal(sixth(m), s)
        # both sides never fall as m grows, so they agree everywhere if they agree
        # wherever either steps, and at the ends
        code = floor_code_of_sixth(m)
        step = np.flatnonzero(np.diff(code))
        assert np.all(np.diff(code)[step] > 0) and len(step) <= 9
        at = np.unique(np.concatenate([[0, len(m) - 1], step, step + 1]))
        assert np.array_equal(code[at], floor_code(s[at])), e


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


CODES = np.array([c * 2.0 ** -9 if c < 8 else (1 + (c & 7) / 8) * 2.0 ** ((c >> 3) - 7) for c in range(127)])


def rn_code(s):
    """E4M3 code nearest s, ties to the even code, at least 1 and at most 126."""
    s = s.astype(np.float64)
    lo = np.clip(np.searchsorted(CODES, s, side="right") - 1, 0, 125)
    mid = (CODES[lo] + CODES[lo + 1]) / 2
    return np.maximum(np.where((s > mid) | ((s == mid) & (lo % 2 == 1)), lo + 1, lo), 1)


@pytest.mark.gpu
@pytest.mark.parametrize("rows", [1, 64])
def test_kernels_against_the_division(rows):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2606_07618_gb300 import binding as B
    rng = np.random.default_rng(rows)
    mids = (CODES[1:] + CODES[:-1]) / 2
    m = np.concatenate([around(CODES[1:]), around(mids), np.float32([1e-30, 5e3, 1e9, 2.0 ** 47])])
    more = (rng.integers(0, 1 << 23, 1 << 15) | (rng.integers(118, 141, 1 << 15) << 23)).astype(np.uint32).view(np.float32)
    m = np.concatenate([m, more])
    m = m[:len(m) // rows * rows]
    x = np.zeros((rows, len(m) // rows, 16), dtype=np.float32)
    where = rng.integers(0, 16, x.shape[:2])
    np.put_along_axis(x, where[..., None], (m * rng.choice([-1.0, 1.0], len(m)).astype(np.float32)).reshape(rows, -1, 1), 2)
    xd = torch.from_numpy(x.reshape(rows, -1)).cuda()
    S = torch.ones(1, device="cuda")                          # y = x
    s = m / np.float32(6)
    for call, want in (("sweep", np.maximum(floor_code(s), 1)), ("absmax", rn_code(s))):
        o = B.empty_outputs(rows, xd.shape[1], 16, linear=True)
        if call == "sweep":
            B.scalesweep_quantize(xd, 16, S, B.NVFP4_OBJ_MSE, None, 0, 0, 0, o["codes"], o["sf_linear"])
        else:
            B.absmax_quantize(xd, 16, S, o["codes"], o["sf_linear"])
        got = o["sf_linear"].cpu().numpy().reshape(-1)
        assert np.array_equal(got, want), (call, m[np.flatnonzero(got != want)[:4]])
