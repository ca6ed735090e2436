"""Raw mode products on buffers off 16 bytes: element-wise kernels where the
library has them, an error before any launch elsewhere."""
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


def _off(n, dtype, bytes_off):
    """A tensor of n elements that starts bytes_off bytes after a 16-byte boundary."""
    k = bytes_off // dtype.itemsize
    t = torch.empty(n + 16, dtype=dtype, device="cuda")
    assert t.data_ptr() % 16 == 0
    v = t[k:k + n]
    assert v.data_ptr() % 16 == bytes_off
    return v


@pytest.mark.parametrize("prec,ns,flags,xo,yo", [("fp64", [40, 24], 1, 8, 0), ("fp64", [40, 24], 0, 8, 8),
                                                 ("fp64", [400, 10], 1, 0, 8), ("bf16x3", [264, 16], 5, 4, 0),
                                                 ("bf16x3", [264, 16], 4, 8, 12), ("bf16x3", [1030, 9], 5, 0, 4),
                                                 ("bf16x3", [264], 4, 4, 4)])
def test_element_aligned(fc, prec, ns, flags, xo, yo):
    d = len(ns)
    s = fc.Solver(ns, [(-4.0, 4.0)] * d, [1.3, 1.7][:d], 1.0, 0.4, 0.5, 1.0, 0.2, precision=prec)
    f64 = prec == "fp64"
    dt, eps, pad = (torch.float64, 2.0 ** -53, 4) if f64 else (torch.float32, 2.0 ** -24, 8)
    p = (ns[0] + pad - 1) // pad * pad
    P = fc.fcgle_internal_elems(s.h)
    R = P // p
    g = torch.Generator(device="cuda").manual_seed(4)
    X0 = torch.randn(2 * R, p, dtype=dt, device="cuda", generator=g)
    X0[:, ns[0]:] = 0.0
    X, Y = _off(2 * P, dt, xo), _off(2 * P, dt, yo)
    X.copy_(X0.reshape(-1))
    A0 = torch.empty(2 * P, dtype=dt, device="cuda")
    fc.fcgle_mode_product(s.h, 0, flags, X0.reshape(-1).contiguous(), A0)
    fc.fcgle_mode_product(s.h, 0, flags, X, Y)
    s.sync()
    # both within p roundings of sum |M| |x| <= |x|_2 (rows of M have norm 1)
    tol = 2 * p * eps * X0.norm(dim=1).max().item()
    assert (A0 - Y).abs().max().item() <= tol
    assert A0.abs().max().item() > 0.1
    s.close()


@pytest.mark.parametrize("prec,ns,flags,xo,yo", [("bf16x3", [40, 24], 0, 4, 0), ("bf16x3", [40, 24], 1, 0, 8),
                                                 ("bf16x3", [40, 24], 5, 4, 0), ("bf16x3", [40, 24], 3, 0, 8)])
def test_refused(fc, prec, ns, flags, xo, yo):
    s = fc.Solver(ns, [(-4.0, 4.0)] * 2, [1.3, 1.7], 1.0, 0.4, 0.5, 1.0, 0.2, precision=prec)
    P = fc.fcgle_internal_elems(s.h)
    X, Y = _off(2 * P, torch.float32, xo), _off(2 * P, torch.float32, yo)
    with pytest.raises(fc.FcgleError) as e:
        fc.fcgle_mode_product(s.h, 0, flags, X, Y)
    assert e.value.status == fc.FCGLE_ERR_INVALID_ARG
    s.close()
