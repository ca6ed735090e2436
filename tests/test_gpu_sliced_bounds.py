"""FP64 sliced products at their bounds and beyond: infinities, and data whose digits are in line with the matrix's, so
that the digit sums come near their bounds, against extended precision.

Tolerance: that of test_gpu_sliced.py (each operand entry cut at 2^-55 of its
row's largest, random over K, times 8, plus the rounding of the result)."""
from fractions import Fraction

import numpy as np
import pytest

from test_slice_segment import _digits

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fc():
    import __graft_entry__ as g
    g.build()
    from paper_2510_21394_gb300 import fcgle
    return fcgle


def _problem(fc, n):
    """FP64 handle of (n, 8), its product of direction 0 on rows (2 R, p), and the matrix M[i][k] read back."""
    s = fc.Solver([n, 8], [(-4.0, 4.0), (-3.0, 3.0)], [1.3, 1.7], 1.0, 0.4, 0.5, 1.0, 0.2, precision="fp64")
    p = (n + 3) // 4 * 4
    R = fc.fcgle_internal_elems(s.h) // p

    def product(X):
        Xd = torch.from_numpy(np.ascontiguousarray(X)).cuda().reshape(-1)
        Y = torch.full_like(Xd, 7.0)
        fc.fcgle_mode_product(s.h, 0, 1, Xd, Y)
        s.sync()
        return Y.reshape(2, p, R).permute(0, 2, 1).reshape(2 * R, p).cpu().numpy()

    cols = []
    for k0 in range(0, p, 2 * R):
        E = np.zeros((2 * R, p))
        m = min(2 * R, p - k0)
        E[np.arange(m), k0 + np.arange(m)] = 1.0
        cols.append(product(E)[:m])
    return s, p, R, product, np.concatenate(cols).T


@pytest.mark.parametrize("n", [1023, 1500])
def test_digits_in_line(fc, n):
    s, p, R, product, M = _problem(fc, n)
    # row r: digits as large as they come and in line with those of row i = i_r of M,
    # digit b with level 4 - b, so that all five products of level 4 have one sign; odd
    # rows: all of one sign
    rows = np.linspace(0, n - 1, 2 * R).astype(int)
    dig = _digits(M[rows])
    X = np.zeros((2 * R, p))
    for r in range(2 * R):
        for b in range(5):
            sgn = np.where(dig[4 - b, r] < 0, -1.0, 1.0) if r % 2 == 0 else np.ones(p)
            X[r] += (127.0 if b else 63.0) * sgn * 2.0 ** (-8 * b)
    X[:, n:] = 0.0
    Y = product(X)
    T = X.astype(np.longdouble) @ M.astype(np.longdouble).T
    err = np.abs(Y.astype(np.longdouble) - T)
    xm = np.abs(X).max(axis=1, keepdims=True).astype(np.longdouble)
    mm = np.abs(M).max(axis=1)[None, :].astype(np.longdouble)
    assert np.all(err <= 2.0 ** -53 * np.abs(T) + 8 * 2.0 ** -55 * np.sqrt(p) * xm * mm)
    s.close()


@pytest.mark.parametrize("n,terms", [(1500, 8), (1500, 40), (400, 8)])
def test_exact_sums_round_once(fc, n, terms):
    """Operands without a cut: data with one digit, matrix entries within 1/4 of
    their row's largest.  The integer sum is then exact, and the result is its
    rounding to 53 bits (through an integer of 62 bits: 2^-53 (1 + 2^-8))."""
    s, p, R, product, M = _problem(fc, n)
    rng = np.random.default_rng(11)
    X = np.zeros((2 * R, p))
    big = np.abs(M) >= np.abs(M).max(axis=1, keepdims=True) / 4
    ok = np.zeros((2 * R, p), bool)
    for r in range(2 * R):
        k = rng.permutation(np.flatnonzero(big[rng.integers(0, n)]))[:terms]   # one output at least qualifies
        X[r, k] = 63.0 / 32.0 * np.where(M[rng.integers(0, n), k] < 0, -1.0, 1.0)
        ok[r] = big[:, k].all(axis=1)
    ok[:, n:] = False
    assert ok.any(axis=1).all()
    Y = product(X)
    for r in range(2 * R):
        k = np.flatnonzero(X[r])
        for i in np.flatnonzero(ok[r])[:40]:
            t = sum(Fraction(float(X[r, c])) * Fraction(float(M[i, c])) for c in k)
            assert abs(Fraction(float(Y[r, i])) - t) <= abs(t) * Fraction(257, 256) / 2 ** 53
    s.close()


@pytest.mark.parametrize("prec,ns", [("fp64", [40, 24]), ("fp64", [134, 9]), ("bf16x3", [264, 16]), ("bf16x3", [1040, 8])])
def test_infinities_keep_their_sign(fc, prec, ns):
    """A row with infinities gives what the sum gives: +-Inf by the matrix entry's
    sign, NaN where infinities of both signs meet or a zero entry does."""
    s = fc.Solver(ns, [(-4.0, 4.0)] * 2, [1.3, 1.7], 1.0, 0.4, 0.5, 1.0, 0.2, precision=prec)
    f64 = prec == "fp64"
    dt, pad = (np.float64, 4) if f64 else (np.float32, 8)
    p = (ns[0] + pad - 1) // pad * pad
    R = fc.fcgle_internal_elems(s.h) // p

    def product(X):
        Xd = torch.from_numpy(np.ascontiguousarray(X)).cuda().reshape(-1)
        Y = torch.full_like(Xd, 7.0)
        fc.fcgle_mode_product(s.h, 0, 1 if f64 else 5, Xd, Y)
        s.sync()
        return Y.reshape(2, p, R).permute(0, 2, 1).reshape(2 * R, p).cpu().numpy()

    cols = []
    for k0 in range(0, p, 2 * R):
        E = np.zeros((2 * R, p), dt)
        m = min(2 * R, p - k0)
        E[np.arange(m), k0 + np.arange(m)] = 1.0
        cols.append(product(E)[:m])
    M = np.concatenate(cols).T
    rng = np.random.default_rng(3)
    X = rng.standard_normal((2 * R, p)).astype(dt)
    X[:, ns[0]:] = 0.0
    want = product(X)
    bad = {2: {5: np.inf}, 3: {7: -np.inf}, 5: {0: np.inf, 9: np.inf}, 6: {1: np.inf, 2: -np.inf},
           2 * R - 1: {ns[0] - 1: np.inf}, 9: {3: np.inf, 4: np.nan}}
    for r, e in bad.items():
        for k, v in e.items():
            X[r, k] = v
        with np.errstate(invalid="ignore"):
            want[r] = sum(M[:, k] * dt(v) for k, v in e.items())
    Y = product(X)
    assert np.array_equal(Y, want, equal_nan=True)
    s.close()
