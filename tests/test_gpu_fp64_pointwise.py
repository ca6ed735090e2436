"""FP64 e^{theta K} v entry by entry, far out in the algebraic tails of the
fractional operator, where the result is many orders below its maximum: no
further from the exponential's power series in extended precision than a plain
FP64 product with the same matrix."""
import math

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


def _D(n, alpha, h):
    g = np.empty(n)
    g[0] = math.gamma(alpha + 1) / math.gamma(alpha / 2 + 1) ** 2
    for k in range(1, n):
        g[k] = (1 - (alpha + 1) / (alpha / 2 + k)) * g[k - 1]
    i = np.arange(n)
    return -h ** (-alpha) * g[np.abs(i[:, None] - i[None, :])]


def _expv(A, z, u):
    """e^{z A} u by its series in np.longdouble, in steps of |z| ||A|| <= 2."""
    A = A.astype(np.longdouble)
    m = max(1, math.ceil(abs(z) * float(np.abs(A).sum(axis=1).max()) / 2))
    v, zc = u.astype(np.clongdouble), np.clongdouble(z) / m
    for _ in range(m):
        t, s = v, v
        for k in range(1, 40):
            t = (A @ t) * (zc / k)
            s = s + t
        v = s
    return v


@pytest.mark.parametrize("n,alpha,box,theta", [(200, 1.5, 10.0, 1e-4), (200, 1.5, 10.0, 1e-3), (160, 1.2, 10.0, 1e-2),
                                               (200, 1.8, 20.0, 1e-3)])
def test_tails_of_the_exponential(fc, n, alpha, box, theta):
    nu, eta = 1.0, 0.5
    h = 2 * box / (n + 1)
    A = _D(n, alpha, h)
    x = -box + h * np.arange(1, n + 1)
    u = np.exp(-x ** 2).astype(np.complex128)
    exact = _expv(A, theta * complex(nu, eta), u)
    s = fc.Solver([n], [(-box, box)], [alpha], nu, eta, 0.0, 1.0, 0.0, precision="fp64")
    # Q of the handle (two unit vectors per product), then the plain FP64 product
    P = fc.fcgle_internal_elems(s.h)
    Q = np.zeros((n, n))
    for k in range(0, n, 2):
        X = torch.zeros(2 * P, dtype=torch.float64, device="cuda")
        X[k] = 1.0
        if k + 1 < n:
            X[P + k + 1] = 1.0
        Y = torch.empty_like(X)
        fc.fcgle_mode_product(s.h, 0, 0, X, Y)
        s.sync()
        Q[:, k:k + 2] = Y.reshape(2, P)[:, :n].T.cpu().numpy()[:, :n - k]
    w = np.einsum("ij,ij->j", Q, A @ Q)
    plain = ((Q * np.exp(theta * complex(nu, eta) * w)) @ Q.T) @ u
    got = s.apply_f("exp", 0, theta, torch.from_numpy(u).cuda())
    s.sync()
    got = got.cpu().numpy()
    s.close()

    def err(y):
        return np.abs(y.astype(np.clongdouble) - exact) / np.abs(exact)
    # one matrix (to its rounding), so one error, up to that of adding in another order
    assert err(got).max() <= 1.25 * err(plain).max()
    assert np.median(err(got)) <= 1.25 * np.median(err(plain))
    nrm = [np.linalg.norm((y.astype(np.clongdouble) - exact).astype(np.complex128)) for y in (got, plain)]
    assert nrm[0] <= 1.25 * nrm[1]
