"""Operands and source terms fetched ahead by the fused-epilogue products
(b3_kernel.cuh), and the adjoint's kept storage.

The ring of a warp holds a few blocks of operand planes; with more source terms
fewer blocks (down to one) and, at four terms, not every term fits.  Each count is
run on both operand forms (p <= 256: M in tensor memory; p > 256: streamed) and
on extents with ragged tiles, against the FP64 oracle at the split-BF16 schemes'
1e-4 (each product about 1e-5)."""
import numpy as np
import pytest

from helpers import PARS, rand_tensor, rel
from oracle import schemes, tensor

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fc():
    import __graft_entry__ as g
    g.build()
    from paper_2510_21394_gb300 import fcgle
    return fcgle


@pytest.mark.parametrize("ns", [[20, 27, 13], [264, 9], [17, 272]])
@pytest.mark.parametrize("scheme", ["lie", "etd2rk", "lbdf2"])
@pytest.mark.parametrize("nsrc", [1, 2, 3, 4])
def test_sources(fc, ns, scheme, nsrc):
    d = len(ns)
    boxes, al = [(-4.0, 4.0), (-3.0, 3.0), (-5.0, 5.0)][:d], [1.5, 1.2, 1.9][:d]
    P = tensor.Problem(ns, boxes, al, *PARS.values())
    sig = [-1.0, 0.5j, -0.3 + 1.0j, 0.2][:nsrc]
    S = [0.5 * rand_tensor(ns, 10 + k) for k in range(nsrc)]
    u0 = rand_tensor(ns, 1)
    ref = schemes.integrate(tensor.Spectral(P), schemes.Nonlinearity(P, sig, S), scheme, 1e-3, 3, u0)
    s = fc.Solver(ns, boxes, al, **PARS, precision="bf16x3")
    s.set_source(sig, [torch.from_numpy(x.astype(np.complex64)).cuda() for x in S])
    got = s.integrate(scheme, 1e-3, 3, torch.from_numpy(u0.astype(np.complex64)).cuda())
    s.sync()
    assert rel(got.cpu().numpy(), ref) <= 1e-4
    s.close()


@pytest.mark.parametrize("prec", ["bf16x3", "fp64"])
def test_adjoint_storage_reuse(fc, prec):
    """Gradients on one handle, the storage kept, grown and used again, equal those of fresh
    handles (bit for bit up to the order of the atomic sums of loss and parameters)."""
    ns, boxes, al = [24, 20, 16], [(-4.0, 4.0), (-3.0, 3.0), (-5.0, 5.0)], [1.5, 1.2, 1.9]
    dt = torch.complex128 if prec == "fp64" else torch.complex64
    u = torch.from_numpy(rand_tensor(ns, 2)).to(dt).cuda()
    t = torch.from_numpy(rand_tensor(ns, 3)).to(dt).cuda()
    one = fc.Solver(ns, boxes, al, **PARS, precision=prec)
    for steps, ck in ((2, 1), (5, 2), (1, 0), (5, 2)):
        a = one.adjoint("lawson_rk2", 1e-3, steps, u, t, ckpt_every=ck)
        fresh = fc.Solver(ns, boxes, al, **PARS, precision=prec)
        b = fresh.adjoint("lawson_rk2", 1e-3, steps, u, t, ckpt_every=ck)
        fresh.close()
        assert torch.equal(a[1], b[1])
        assert a[0] == pytest.approx(b[0], rel=1e-12)
        assert np.allclose(a[2], b[2], rtol=1e-9, atol=1e-9 * max(abs(x) for x in b[2]))
    one.close()
