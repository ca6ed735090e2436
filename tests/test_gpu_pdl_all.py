"""Dependent launch of the slicing, layout, pointwise and adjoint kernels: the
same bits with FCGLE_PDL=0 (plain launches) as with the default, on the paths
of FP64 handles, of extents above 256, of the adjoint and of sources.  The
library reads the switch once per process, so each setting runs in its own."""
import os
import subprocess
import sys

import numpy as np
import pytest

pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

RUN = r"""
import sys
import numpy as np
import torch
sys.path.insert(0, sys.argv[1])
from paper_2510_21394_gb300 import fcgle, inputs

out = {}
def run(name, ns, prec, scheme, steps, source=False, form=None):
    dt = torch.complex128 if prec == "fp64" else torch.complex64
    boxes = [(-6.0, 6.0)] * len(ns)
    u0 = torch.from_numpy(inputs.gaussian_random_phase(ns, boxes, seed=3)).to(dt).cuda()
    s = fcgle.Solver(ns, boxes, [1.3, 1.5, 1.7][:len(ns)], nu=1.0, eta=0.5, gamma=1.0, kappa=1.0, zeta=0.5, precision=prec)
    if source:
        s.set_source([-1.0, 0.5j], [(0.1 * u0).contiguous(), (0.2j * u0).contiguous()])
    if form:
        s.set_exp_form(form)
    for k in range(3):   # back to back, so that launches overlap from call to call
        y = s.integrate(scheme, 1e-3, steps, u0)
    z = s.apply_f("phi", 2, 1e-2, y)
    out[name] = y
    out[name + "_f"] = z
    if len(ns) == 3 and prec == "bf16x3":
        loss, grad, gp = s.adjoint("lawson_rk2", 1e-3, 4, u0, (0.9 * u0).contiguous(), ckpt_every=2)
        out["adj_" + name] = grad
        out["sum_" + name] = torch.tensor([loss] + list(gp), dtype=torch.float64)
    torch.cuda.synchronize()
    s.close()

run("a", [60, 44, 28], "fp64", "krogstad", 4)
run("b", [300, 68], "fp64", "lbdf2", 6, source=True)
run("c", [90, 64], "fp64", "strang", 4)
run("d", [300, 264], "bf16x3", "etd2rk", 6)
run("e", [272, 16, 24], "bf16x3", "lbdf2", 5, source=True)
run("f", [64, 48, 40], "bf16x3", "strang", 5)
run("g", [64, 40], "bf16x3", "lawson_rk2", 5, source=True, form="kron")
np.savez(sys.argv[2], **{k: v.cpu().numpy() for k, v in out.items()})
"""


def _run(tmp_path, pdl):
    env = dict(os.environ)
    env.pop("FCGLE_PDL", None)
    if pdl:
        env["FCGLE_PDL"] = pdl
    path = str(tmp_path / ("pdl_%s.npz" % pdl))
    subprocess.run([sys.executable, "-c", RUN, ROOT, path], env=env, check=True, timeout=600)
    with np.load(path) as z:
        return {k: z[k] for k in z.files}


def test_same_bits_without_dependent_launch(tmp_path):
    import __graft_entry__ as g
    g.build()
    on, off = _run(tmp_path, None), _run(tmp_path, "0")
    assert on.keys() == off.keys() and len(on) == 18
    for k in on:
        assert np.isfinite(on[k]).all(), k
        if k.startswith("sum_"):
            # sums by FP64 atomics, in any order over at most 2^17 terms: 2^17 2^-53 of their magnitude
            assert np.all(np.abs(on[k] - off[k]) <= 2.0 ** -36 * np.abs(off[k]).max()), k
        else:
            assert np.array_equal(on[k], off[k]), k
