"""The phi polynomial along the ray z = theta (nu + i eta) s at any size of
theta (nu + i eta): its coefficients stay in the range of FP32."""
import numpy as np
import pytest

from helpers import rel_norm
from oracle import phi as ophi
from test_gpu_numeric import TOL32

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fc():
    import __graft_entry__ as g
    g.build()
    from paper_2510_21394_gb300 import fcgle
    return fcgle


@pytest.mark.parametrize("w", [1e-20, 1e-9, 1e-7, 1e-6, 1e-5, 1e-3, 1.0, 1e3, 1e6, 1e9, 1e20])
@pytest.mark.parametrize("k", [1, 2, 3])
def test_ray_polynomial_at_any_scale(fc, w, k):
    theta = 1e-3
    nu, eta = w / theta, 0.5 * w / theta
    s = fc.Solver([7, 9], [(-1.0, 1.0), (-3.0, 2.0)], [1.2, 1.8], nu, eta, 0.5, 1.0, 0.2, precision="bf16x3")
    z = np.concatenate([[0.0], np.logspace(-6, -0.001, 60), [1.01, 2.0, 4.5]])
    sv = (-z / (w * abs(1 + 0.5j))).astype(np.float32).astype(np.float64)
    got = np.array(fc.fcgle_spectral_scalars(s.h, "phi", k, theta, sv, 1))
    ref = ophi.phi(k, theta * complex(nu, eta) * sv)
    # the bounds of the unit-sized case (test_gpu_numeric.py)
    assert np.all(np.abs(got - ref) <= TOL32[k] * np.abs(ref))
    s.close()


@pytest.mark.parametrize("scheme", ["lawson_euler", "lawson_rk2", "strang", "etd2rk"])
@pytest.mark.parametrize("scale", [1e-7, 1e8])
def test_schemes_in_other_units(fc, scheme, scale):
    """Lengths in other units: the same spectrum from a diffusion coefficient of
    another size, the same states to the rounding of the precision."""
    ns, al = [40, 36], 1.5
    tau, steps = 1e-2, 5
    out = []
    for nu, L in ((1.0, 1.0), (scale, scale ** (1.0 / al))):   # nu h^-alpha is the same
        s = fc.Solver(ns, [(-6.0 * L, 6.0 * L)] * 2, [al, al], nu, 0.5 * nu, 0.5, 1.0, 0.2, precision="bf16x3")
        x = np.linspace(-6, 6, ns[0] + 2)[1:-1][None, :]
        y = np.linspace(-6, 6, ns[1] + 2)[1:-1][:, None]
        u = torch.from_numpy(np.exp(-x ** 2 - y ** 2) * (1 + 0.3j * x)).to(torch.complex64).cuda()
        o = s.integrate(scheme, tau, steps, u)
        s.sync()
        out.append(o.cpu().numpy())
        s.close()
    # at most 4 Tucker operators per step and run, 1e-5 each
    assert np.isfinite(out[1]).all() and rel_norm(out[1], out[0]) <= 2 * steps * 4 * 1e-5
