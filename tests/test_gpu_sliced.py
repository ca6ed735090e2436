"""Sliced mode products (FP64 handles, precise FP32 products with p > 256)
against extended precision on the host.

The matrix is read back through unit rows; the data rows span magnitudes from
1e-250 to 1e250 (FP64) or 1e-30 to 1e30 (FP32), with a constant row
(all digits coherent), a zero row and a last row whose entries fall off by many
orders.

Tolerance per entry, from the slicing (sliced.cu): every operand entry is cut at
half a unit, at most 2^-55 (FP64) or 2^-26 (FP32) of its row's largest entry,
and the dropped levels lie below that, so over K entries the error is a random
sum of standard deviation about 2^-55 sqrt(K) max|x| max|M_i| (2^-26 for FP32);
8 of them, plus the rounding of the result (and of the FP32 accumulator above
2^24: two more)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fc():
    import __graft_entry__ as g
    g.build()
    from paper_2510_21394_gb300 import fcgle
    return fcgle


# p_1 at the edges of the 32-wide chunks, the 64-wide and 128-wide matrix tiles and the range;
# 2 R around the 128-row tiles and far below them
SHAPES64 = [[200], [132, 3], [16, 9], [20, 8], [31, 64], [64, 65], [66, 33], [130, 6, 5], [256, 63], [1000, 70], [1024, 20], [1028, 8]]
SHAPES32 = [[257, 64], [272, 9], [512, 65], [1017, 40], [1024, 24], [1025, 16]]


def _rows(R2, p, n, dt, seed):
    rng = np.random.default_rng(seed)
    X = rng.standard_normal((R2, p))
    X[:, n:] = 0.0
    big = 250.0 if dt == np.float64 else 30.0
    X *= 10.0 ** rng.uniform(-big, big, (R2, 1))
    X[0, :n] = 1.0 / 3.0
    X[1] = 0.0
    X[R2 - 1, :n] = np.exp(-np.linspace(0.0, 60.0, n))
    return X.astype(dt)


@pytest.mark.parametrize("prec,ns", [("fp64", ns) for ns in SHAPES64] + [("bf16x3", ns) for ns in SHAPES32])
@pytest.mark.parametrize("fwd", [0, 1])
def test_sliced_product(fc, prec, ns, fwd):
    d = len(ns)
    s = fc.Solver(ns, [(-4.0, 4.0), (-3.0, 3.0), (-5.0, 5.0)][:d], [1.3, 1.7, 1.5][:d], 1.0, 0.4, 0.5, 1.0, 0.2,
                  precision=prec)
    f64 = prec == "fp64"
    dt, tdt, pad, flags = (np.float64, torch.float64, 4, fwd) if f64 else (np.float32, torch.float32, 8, fwd | 4)
    n, p = ns[0], (ns[0] + pad - 1) // pad * pad
    R = fc.fcgle_internal_elems(s.h) // p

    def product(X):
        Xd = torch.from_numpy(np.ascontiguousarray(X)).cuda().reshape(-1)
        Y = torch.full_like(Xd, 7.0)
        fc.fcgle_mode_product(s.h, 0, flags, Xd, Y)
        s.sync()
        return Y.reshape(2, p, R).permute(0, 2, 1).reshape(2 * R, p).cpu().numpy()

    cols = []
    for k0 in range(0, p, 2 * R):
        E = np.zeros((2 * R, p), dt)
        m = min(2 * R, p - k0)
        E[np.arange(m), k0 + np.arange(m)] = 1.0
        cols.append(product(E)[:m])
    M = np.concatenate(cols).T                      # M[i][k]
    X = _rows(2 * R, p, n, dt, 5)
    Y = product(X)
    # np.longdouble on sampled rows (64 or more mantissa bits)
    rows = np.unique(np.concatenate([np.arange(min(3, 2 * R)), np.linspace(0, 2 * R - 1, 24).astype(int)]))
    T = X[rows].astype(np.longdouble) @ M.astype(np.longdouble).T
    err = np.abs(Y[rows].astype(np.longdouble) - T)
    xm = np.abs(X[rows]).max(axis=1, keepdims=True).astype(np.longdouble)
    mm = np.abs(M).max(axis=1)[None, :].astype(np.longdouble)
    u, cut = (2.0 ** -53, 2.0 ** -55) if f64 else (3 * 2.0 ** -24, 2.0 ** -26)
    tiny = np.finfo(dt).tiny
    assert np.all(err <= u * np.abs(T) + 8 * cut * np.sqrt(p) * xm * mm + tiny)
    assert np.all(Y[:, n:] == 0.0)                  # padded output indices stay zero
    assert 2 * R == 2 or np.all(Y[1] == 0.0)
    s.close()


@pytest.mark.parametrize("prec,ns", [("fp64", [40, 24]), ("bf16x3", [264, 16])])
@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
def test_nonfinite_rows(fc, prec, ns, bad):
    """A NaN or an Inf makes exactly its own row of the result non-finite."""
    s = fc.Solver(ns, [(-4.0, 4.0)] * 2, [1.3, 1.7], 1.0, 0.4, 0.5, 1.0, 0.2, precision=prec)
    f64 = prec == "fp64"
    p = ns[0]
    R = fc.fcgle_internal_elems(s.h) // p
    X = _rows(2 * R, p, p, np.float64 if f64 else np.float32, 7)
    X[5, 11] = bad
    Xd = torch.from_numpy(X).cuda().reshape(-1)
    Y = torch.zeros_like(Xd)
    fc.fcgle_mode_product(s.h, 0, 1 if f64 else 5, Xd, Y)
    s.sync()
    Yr = Y.reshape(2, p, R).permute(0, 2, 1).reshape(2 * R, p).cpu().numpy()
    fin = np.isfinite(Yr)
    assert not fin[5].any() and fin[np.arange(2 * R) != 5].all()
    s.close()


@pytest.mark.parametrize("ns", [[20, 36], [520, 16], [33, 20, 29]])
def test_complex_block_form(fc, ns):
    """FP64 e^{theta K} v by the Kronecker-product form: contractions of 2 p over both planes."""
    from helpers import PARS, rand_tensor, rel
    from oracle import tensor
    d = len(ns)
    boxes, al = [(-4.0, 4.0), (-3.0, 3.0), (-5.0, 5.0)][:d], [1.5, 1.2, 1.9][:d]
    v = rand_tensor(ns, 3)
    s = fc.Solver(ns, boxes, al, **PARS, precision="fp64")
    got = s.apply_f("exp", 0, 1e-2, torch.from_numpy(v).cuda())
    s.sync()
    ref = tensor.Spectral(tensor.Problem(ns, boxes, al, *PARS.values())).apply_f("exp", 0, 1e-2, v)
    assert rel(got.cpu().numpy(), ref) <= 1e-12
    s.close()
