"""Segments of the FP64 sliced products (host side): with the data's digits at
their largest and in line with the matrix's, the leading digit sums of every
segment stay within the 2^24 that an FP32 accumulator holds exactly, and no
longer segment would do."""
import math

import numpy as np
import pytest


def _digits(M):
    """Balanced digits of every entry, 8 of 8 bits, one exponent per row (python integers)."""
    out = np.zeros((8,) + M.shape, dtype=np.int64)
    off = sum(1 << (8 * j + 7) for j in range(7))
    for i, row in enumerate(M):
        top = np.max(np.abs(row))
        if top == 0.0:
            w = [off] * row.size
        else:
            e = math.frexp(top)[1]
            # 62 bits below the leading power of two, half away from zero (integer arithmetic:
            # 62 bits do not fit a double)
            w = []
            for x in row:
                m, ex = math.frexp(x)
                n, sh = int(math.ldexp(abs(m), 53)), 62 - 53 - (e - ex)
                n = n << sh if sh >= 0 else (n + (1 << (-sh - 1))) >> -sh
                w.append((n if x >= 0 else -n) + off)
        for a in range(8):
            out[a, i] = [v >> 56 if a == 0 else ((v >> (8 * (7 - a))) & 255) - 128 for v in w]
    return out


def _level(dig, seg):
    """The largest |P_0| .. |P_4| any data can give: all partners at their largest (128, the
    top digit 64) and in line."""
    s = 128 * np.abs(dig[:4]).sum(axis=0) + 64 * np.abs(dig[4])
    return max(int(s[:, k:k + seg].sum(axis=1).max()) for k in range(0, s.shape[1], seg))


def _Q(n, alpha):
    g = np.empty(n)
    g[0] = math.gamma(alpha + 1) / math.gamma(alpha / 2 + 1) ** 2
    for k in range(1, n):
        g[k] = (1 - (alpha + 1) / (alpha / 2 + k)) * g[k - 1]
    i = np.arange(n)
    return np.linalg.eigh(-g[np.abs(i[:, None] - i[None, :])])[1]


CASES = {
    "constant": lambda: np.full((3, 1024), 0.995),
    "digits_in_line": lambda: np.full((2, 1000), sum(127.0 * 256.0 ** -a for a in range(1, 5))),
    "zero_row": lambda: np.vstack([np.zeros(96), np.ones(96)]),
    "short": lambda: np.random.default_rng(1).standard_normal((40, 40)),
    "Q400": lambda: _Q(400, 1.5),
    "Q1023T": lambda: _Q(1023, 1.3).T.copy(),
    "graded": lambda: np.exp(-np.abs(np.arange(600)[:, None] - np.arange(600)[None, :]) / 9.0),
}


@pytest.mark.parametrize("name", CASES)
def test_leading_levels_fit(name):
    from paper_2510_21394_gb300 import fcgle
    M = CASES[name]()
    K = M.shape[1]
    seg = fcgle.fcgle_selftest_slice_segment(M)
    chunks = (K + 31) // 32
    assert seg % 32 == 0 and 0 < seg <= 32 * chunks
    dig = _digits(M)
    assert _level(dig, seg) <= 1 << 24
    n = -(-chunks // (seg // 32))
    if n > 1:   # one segment less is too long
        longer = 32 * -(-chunks // (n - 1))
        assert longer > 1024 or _level(dig, longer) > 1 << 24


def test_constant_row_needs_shorter_segments_than_1024():
    from paper_2510_21394_gb300 import fcgle
    assert fcgle.fcgle_selftest_slice_segment(np.full((1, 1024), 0.995)) < 1024
    assert fcgle.fcgle_selftest_slice_segment(_Q(400, 1.5)) >= 400   # and eigenvector matrices of 400 do not
