"""Grouped launches whose instances differ in everything the phi polynomials depend
on: every scheme with one gives the bits of single runs, with more units than
CTAs, so that a CTA meets several instances, and with an instance of one tile."""
import numpy as np
import pytest

from paper_2510_21394_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fc():
    import __graft_entry__ as g
    g.build()
    from paper_2510_21394_gb300 import fcgle
    return fcgle


@pytest.mark.parametrize("scheme", ["lie", "lawson_euler", "lawson_rk2", "etd2rk", "krogstad", "strang"])
def test_grouped_equals_single(fc, scheme):
    rng = np.random.default_rng(8)
    shapes = [[8, 8], [300, 264], [129, 40], [24, 17, 33], [64, 130], [40, 40, 40], [200, 300]]
    specs = [dict(ns=n, boxes=[(-10.0, 10.0)] * len(n), alphas=list(rng.uniform(1.1, 1.9, len(n))),
                  nu=float(rng.uniform(0.3, 2)), eta=float(rng.uniform(-1, 1)), gamma=float(rng.uniform(0, 1)),
                  kappa=float(rng.uniform(0.5, 2)), zeta=float(rng.uniform(-1, 1))) for n in shapes]
    u0 = [torch.from_numpy(inputs.gaussian_pulse(n, [(-3.0, 3.0)] * len(n))).to(torch.complex64).cuda() for n in shapes]
    b = fc.Batch(specs, precision="bf16x3", nstreams=3)
    outs = b.integrate(scheme, 2e-2, 4, u0, grouped=True)
    torch.cuda.synchronize()
    for sp, u, o in zip(specs, u0, outs):
        s = fc.Solver(sp["ns"], sp["boxes"], sp["alphas"], sp["nu"], sp["eta"], sp["gamma"], sp["kappa"], sp["zeta"],
                      precision="bf16x3")
        s.set_tucker_form("rotating")
        ref = s.integrate(scheme, 2e-2, 4, u)
        torch.cuda.synchronize()
        assert torch.isfinite(torch.view_as_real(o)).all() and torch.equal(o, ref), sp["ns"]
        s.close()
    b.close()
