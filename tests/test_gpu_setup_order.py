"""Setup data is ordered on the handle's own stream: FP64 instances made on the
non-blocking streams of a batch, their matrices sliced right after the upload,
give the bits of a handle on the default stream."""
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


def test_fp64_batch_setup_equals_single(fc):
    ns, boxes, al = [300, 212], [(-10.0, 10.0)] * 2, [1.3, 1.7]   # matrices of 720 and 360 KB
    spec = dict(ns=ns, boxes=boxes, alphas=al, nu=1.0, eta=0.5, gamma=1.0, kappa=1.0, zeta=0.5)
    u = torch.from_numpy(inputs.gaussian_pulse(ns, [(-3.0, 3.0)] * 2)).to(torch.complex128).cuda()
    s = fc.Solver(ns, boxes, al, 1.0, 0.5, 1.0, 1.0, 0.5, precision="fp64")
    want = s.integrate("lie", 1e-3, 2, u)
    s.sync()
    s.close()
    for _ in range(3):
        b = fc.Batch([spec] * 6, precision="fp64", nstreams=6)
        outs = b.integrate("lie", 1e-3, 2, [u] * 6)
        torch.cuda.synchronize()
        for o in outs:
            assert torch.equal(o, want)
        b.close()
