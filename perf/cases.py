"""Performance cases of the FCGLE time-stepping library.

Each case is one call (or one short integration) a program makes through the
public binding ``paper_2510_21394_gb300.fcgle``: ``Solver.apply_f``,
``Solver.integrate``, ``Solver.adjoint`` and ``Batch.integrate``, in both
precisions, from a 64 x 64 grid to 425^3.  ``prepare`` makes what such a
program has in hand (a solver handle and device tensors), ``run`` makes the
call, ``exact`` evaluates the same result with plain torch in complex128.
"""
import math

import numpy as np
import torch

SCHEMES = ("lie", "lawson_euler", "lawson_rk2", "etd2rk", "krogstad", "lbdf2", "strang")
ALPHAS = {1: (1.5,), 2: (1.3, 1.7), 3: (1.2, 1.5, 1.8)}
COEFFS = (1.0, 0.5, 1.0, 1.0, 0.5)   # nu, eta, gamma, kappa, zeta


def listed():
    return [
        # the smallest problem a user runs: a 64 x 64 manufactured-solution check, where launches count
        dict(name="small_2d", kind="integrate", prec="bf16x3", ns="64x64", scheme="lawson_euler", steps=10, tau=0.01,
             source=2, box=10.0),
        # one matrix function applied to one field: the building block a user composes own schemes from, 2D
        dict(name="apply_2d", kind="apply", prec="bf16x3", ns="1023x1024", func="phi", k=1, theta=1e-3, box=20.0),
        # the same in 3D on a grid that is ragged in every direction (a resolvent solve)
        dict(name="apply_3d", kind="apply", prec="bf16x3", ns="225x250x199", func="inv", k=0, theta=1e-3, box=10.0),
        # a large 2D pulse run between two outputs of a monitor
        dict(name="etd2rk_2d", kind="integrate", prec="bf16x3", ns="1023x1024", scheme="etd2rk", steps=10, tau=1e-3,
             source=0, box=20.0),
        # the headline 3D run, a stretch of it between two outputs
        dict(name="krogstad_3d", kind="integrate", prec="bf16x3", ns="256x256x256", scheme="krogstad", steps=5,
             tau=1e-3, source=0, box=10.0),
        # Strang splitting at the paper's smallest 3D size
        dict(name="strang_3d", kind="integrate", prec="bf16x3", ns="250x250x250", scheme="strang", steps=5, tau=1e-2,
             source=0, box=10.0),
        # the paper's largest 3D size, linearised BDF2 with a source term: extents above 256
        dict(name="lbdf2_3d_large", kind="integrate", prec="bf16x3", ns="425x425x425", scheme="lbdf2", steps=3,
             tau=1e-2, source=1, box=1.0),
        # a parameter sweep: many uneven instances advanced together
        dict(name="batch_uneven", kind="batch", prec="bf16x3", n2="136 767 301 440 612 188 523 256 371 694 229",
             n3="48 133 160 97 120", scheme="etd2rk", steps=10, tau=1e-3),
        # one gradient evaluation of a parameter and initial-state fit: forward and backward sweep
        dict(name="adjoint_3d", kind="adjoint", prec="bf16x3", ns="128x128x128", steps=10, ckpt=5, tau=1e-3, box=10.0),
        # Kronecker-product form of the exponential, different extents per direction
        dict(name="kron_3d", kind="integrate", prec="bf16x3", ns="256x200x120", scheme="lawson_euler", steps=5,
             tau=1e-3, source=0, box=10.0, form="kron"),
        # the paper's 2D accuracy experiment: double precision, manufactured source, 15 steps
        dict(name="fp64_lbdf2_2d", kind="integrate", prec="fp64", ns="400x400", scheme="lbdf2", steps=15, tau=0.02,
             source=1, box=1.0),
        # double precision in 3D: the run a reduced-precision result is checked against
        dict(name="fp64_krogstad_3d", kind="integrate", prec="fp64", ns="128x120x136", scheme="krogstad", steps=1,
             tau=1e-3, source=0, box=10.0),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _sizes(rng, d, lo, hi, most):
    while True:
        ns = [_log_int(rng, lo, hi) for _ in range(d)]
        if math.prod(ns) <= most:
            return ns


def _text(ns):
    return "x".join(str(n) for n in ns)


def _ns(case):
    return [int(n) for n in case["ns"].split("x")]


def draw(rng):
    kind = rng.choice(["apply", "apply", "integrate", "integrate", "integrate", "fp64", "fp64", "batch", "adjoint", "kron"])
    d = rng.choice([2, 3])
    if kind == "batch":
        return dict(kind="batch", prec="bf16x3", n2=" ".join(str(rng.randint(128, 768)) for _ in range(rng.randint(4, 10))),
                    n3=" ".join(str(rng.randint(48, 160)) for _ in range(rng.randint(1, 4))),
                    scheme=rng.choice(["etd2rk", "krogstad", "lie"]), steps=rng.randint(2, 8), tau=1e-3)
    if kind == "fp64":
        ns = _sizes(rng, d, *((64, 500, 250_000) if d == 2 else (24, 150, 2_000_000)))
        if rng.random() < 0.4:
            func, k = rng.choice([("inv", 0), ("exp", 0), ("phi", rng.randint(1, 4))])
            return dict(kind="apply", prec="fp64", ns=_text(ns), func=func, k=k, theta=rng.choice([1e-3, 1e-2]), box=10.0)
        return dict(kind="integrate", prec="fp64", ns=_text(ns), scheme=rng.choice(SCHEMES), steps=1, tau=1e-3,
                    source=rng.randint(0, 2), box=10.0)
    ns = _sizes(rng, d, *((48, 1100, 1_200_000) if d == 2 else (32, 320, 17_000_000)))
    if kind == "apply":
        func, k = rng.choice([("inv", 0), ("exp", 0), ("phi", rng.randint(1, 4))])
        return dict(kind="apply", prec="bf16x3", ns=_text(ns), func=func, k=k, theta=rng.choice([1e-3, 1e-2]), box=10.0)
    if kind == "adjoint":
        ns = _sizes(rng, d, *((48, 600, 300_000) if d == 2 else (32, 140, 2_200_000)))
        steps = rng.randint(2, 8)
        return dict(kind="adjoint", prec="bf16x3", ns=_text(ns), steps=steps, ckpt=rng.randint(1, steps), tau=1e-3, box=10.0)
    if kind == "kron":
        return dict(kind="integrate", prec="bf16x3", ns=_text(ns), scheme=rng.choice(["lawson_euler", "lawson_rk2", "strang"]),
                    steps=rng.randint(1, 6), tau=1e-3, source=0, box=10.0, form="kron")
    return dict(kind="integrate", prec="bf16x3", ns=_text(ns), scheme=rng.choice(SCHEMES), steps=rng.randint(1, 8), tau=1e-3,
                source=rng.randint(0, 2), box=10.0)


# ------------------------------------------------------------------ inputs
def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _coords(ns, box, dev):
    """x_mu broadcastable against the tensor shape (n_d, ..., n_1)."""
    d, out = len(ns), []
    for mu, n in enumerate(ns):
        h = 2.0 * box / (n + 1)
        shp = [1] * d
        shp[d - 1 - mu] = n
        out.append((-box + h * torch.arange(1, n + 1, dtype=torch.float64, device=dev)).reshape(shp))
    return out


def _field(ns, box, seed, dev):
    """A localised pulse with a smooth random phase and a little noise (complex128)."""
    rng = np.random.default_rng(seed)
    X = _coords(ns, box, dev)
    w = 1.0 if box > 2.0 else 0.45   # pulse width: well inside the box
    amp, phase = 1.0, 0.0
    for x in X:
        amp = amp * torch.exp(-(x / w) ** 2)
    for _ in range(4):
        t = 0.8 * rng.standard_normal()
        for x in X:
            t = t * torch.cos(rng.uniform(0.3, 1.6) * x / w + rng.uniform(0.0, 2.0 * math.pi))
        phase = phase + t
    g = torch.Generator(device=dev)
    g.manual_seed(int(seed) & 0x7FFFFFFF)
    shape = tuple(reversed(ns))
    noise = torch.randn(shape + (2,), generator=g, device=dev, dtype=torch.float32).double() * 1e-3
    return amp * torch.complex(torch.cos(math.pi * phase), torch.sin(math.pi * phase)) + torch.view_as_complex(noise)


def _source(ns, box, nterms, dev):
    """Source terms e^{sigma_k t} S_k of a decaying (two terms) or an oscillating (one) pulse."""
    if nterms == 0:
        return [], []
    X = _coords(ns, box, dev)
    w = 1.0 if box > 2.0 else 0.45
    G = 1.0
    for x in X:
        G = G * torch.exp(-(x / w) ** 2)
    S1 = G * (-(2.0 + 2.0j) + (0.7 - 0.4j) * X[0])
    if nterms == 1:
        return [-1j], [S1]
    return [-1.0, -3.0], [S1, (1.0 + 3.0j) * G ** 3]


def _dtype(case):
    return torch.complex128 if case["prec"] == "fp64" else torch.complex64


def _specs(case):
    """The instances of a batch: square 2D and cubic 3D grids, coefficients varying from one to the next."""
    out = []
    for j, (d, n) in enumerate([(2, int(n)) for n in case["n2"].split()] + [(3, int(n)) for n in case["n3"].split()]):
        alphas = [1.1 + 0.8 * ((0.37 * j + 0.29 * mu) % 1.0) for mu in range(d)]
        out.append(dict(ns=[n] * d, boxes=[(-10.0, 10.0)] * d, alphas=alphas,
                        nu=0.5 + 0.09 * (j % 16), eta=-1.0 + 0.13 * (j % 16), gamma=0.06 * (j % 16),
                        kappa=0.5 + 0.09 * (j % 13), zeta=1.0 - 0.17 * (j % 12)))
    return out


def _u0(case, seed, dev):
    if case["kind"] == "batch":
        return [_field(sp["ns"], 10.0, seed * 1000 + j, dev).to(_dtype(case)) for j, sp in enumerate(_specs(case))]
    return _field(_ns(case), case["box"], seed, dev).to(_dtype(case))


def _target(case, u0):
    """A state near u(T): the initial state damped and turned."""
    return (u0 * (0.9 - 0.1j)).contiguous()


def prepare(case, seed):
    from paper_2510_21394_gb300 import fcgle

    dev = torch.device("cuda")
    st = dict(case=case)
    if case["kind"] == "batch":
        st["u0"] = _u0(case, seed, dev)
        torch.cuda.synchronize()
        st["batch"] = fcgle.Batch(_specs(case), precision=case["prec"])
        return st
    ns, box, d = _ns(case), case["box"], len(_ns(case))
    st["u0"] = _u0(case, seed, dev)
    s = fcgle.Solver(ns, [(-box, box)] * d, list(ALPHAS[d]), *COEFFS, precision=case["prec"])
    if case.get("source"):
        sig, S = _source(ns, box, case["source"], dev)
        s.set_source(sig, [x.to(_dtype(case)).contiguous() for x in S])
        torch.cuda.synchronize()
    if case.get("form"):
        s.set_exp_form(case["form"])
    if case["kind"] == "adjoint":
        st["target"] = _target(case, st["u0"])
    st["solver"] = s
    return st


def run(state):
    c = state["case"]
    if c["kind"] == "apply":
        return state["solver"].apply_f(c["func"], c["k"], c["theta"], state["u0"])
    if c["kind"] == "integrate":
        return state["solver"].integrate(c["scheme"], c["tau"], c["steps"], state["u0"])
    if c["kind"] == "batch":
        return state["batch"].integrate(c["scheme"], c["tau"], c["steps"], state["u0"], grouped=True)
    loss, grad, gp = state["solver"].adjoint("lawson_rk2", c["tau"], c["steps"], state["u0"], state["target"],
                                             ckpt_every=c["ckpt"])
    return dict(loss=loss, grad_u0=grad, grad_params=torch.tensor(gp, dtype=torch.float64))


# -------------------------------------------------------------------- work
# Tucker operators (2 of them = one f(theta K)) per step of a scheme
_OPS = {"lie": 2, "lawson_euler": 2, "lawson_rk2": 4, "etd2rk": 4, "krogstad": 8, "lbdf2": 2, "strang": 2}


def _flops(ns, ops):
    """ops Tucker operators of real d-mode products on a complex tensor (4 n_mu N each)."""
    return ops * 4.0 * sum(ns) * math.prod(ns)


def work(case):
    el = 16 if case["prec"] == "fp64" else 8
    if case["kind"] == "batch":
        all_ns = [sp["ns"] for sp in _specs(case)]
        return dict(bytes=sum(2 * el * math.prod(n) for n in all_ns),
                    flops=sum(case["steps"] * _flops(n, _OPS[case["scheme"]]) for n in all_ns))
    ns = _ns(case)
    N = math.prod(ns)
    if case["kind"] == "apply":
        return dict(bytes=2 * el * N, flops=_flops(ns, 2))
    if case["kind"] == "adjoint":
        # forward sweep (4 operators a step) and backward sweep (4 a step), end transforms
        return dict(bytes=3 * el * N, flops=_flops(ns, 8 * case["steps"] + 4))
    ops = case["steps"] * _OPS[case["scheme"]]
    return dict(bytes=(2 + case["source"]) * el * N, flops=_flops(ns, ops))


# ------------------------------------------------------- exact (complex128)
class _Exact:
    """K = (nu + i eta) (D_1 (+) ... (+) D_d) through the eigenvectors of its symmetric Toeplitz factors."""

    def __init__(self, ns, boxes, alphas, nu, eta, gamma, kappa, zeta, dev, sigmas=(), S=()):
        self.ns, self.dev, self.S, self.sig = ns, dev, list(S), [complex(s) for s in sigmas]
        self.nu, self.eta, self.gamma, self.kappa, self.zeta = nu, eta, gamma, kappa, zeta
        self.Q, lam = [], 0.0
        for mu, n in enumerate(ns):
            a, (lo, hi) = alphas[mu], boxes[mu]
            g = np.empty(n)
            g[0] = math.gamma(a + 1.0) / math.gamma(a / 2.0 + 1.0) ** 2
            for k in range(1, n):
                g[k] = (1.0 - (a + 1.0) / (a / 2.0 + k)) * g[k - 1]
            i = np.arange(n)
            D = -((hi - lo) / (n + 1)) ** (-a) * g[np.abs(i[:, None] - i[None, :])]
            w, Q = np.linalg.eigh(D)
            self.Q.append(torch.from_numpy(np.ascontiguousarray(Q)).to(dev))
            shp = [1] * len(ns)
            shp[len(ns) - 1 - mu] = n
            lam = lam + torch.from_numpy(w).to(dev).reshape(shp)
        self.lam = lam   # real eigenvalue sums

    @property
    def Lam(self):
        return torch.complex(self.nu * self.lam, self.eta * self.lam)

    def _modes(self, X, Ms):
        d = len(self.ns)
        re, im = X.real, X.imag
        for mu, M in enumerate(Ms):
            ax = d - 1 - mu
            re = torch.movedim(torch.tensordot(re, M, dims=([ax], [1])), -1, ax)
            im = torch.movedim(torch.tensordot(im, M, dims=([ax], [1])), -1, ax)
        return torch.complex(re.contiguous(), im.contiguous())

    def fwd(self, X):
        return self._modes(X, [Q.T for Q in self.Q])

    def bwd(self, X):
        return self._modes(X, self.Q)

    def f(self, func, k, theta):
        z = theta * self.Lam
        if func == "inv":
            return 1.0 / (1.0 - z)
        if func == "exp" or k == 0:
            return torch.exp(z)
        small = z.abs() < 1.0
        zs = torch.where(small, z, torch.zeros_like(z))
        term = torch.full_like(z, 1.0 / math.factorial(k))
        ser = term.clone()
        for m in range(1, 24):
            term = term * zs / (m + k)
            ser = ser + term
        zl = torch.where(small, torch.ones_like(z), z)
        rec = torch.exp(zl)
        for j in range(1, k + 1):
            rec = (rec - 1.0 / math.factorial(j - 1)) / zl
        return torch.where(small, ser, rec)

    def apply(self, func, k, theta, v):
        return self.bwd(self.f(func, k, theta) * self.fwd(v))

    def g(self, t, u):
        r = self.gamma * u - (self.kappa + 1j * self.zeta) * (u.real ** 2 + u.imag ** 2) * u
        for s, S in zip(self.sig, self.S):
            r = r + complex(np.exp(s * t)) * S
        return r

    def flow(self, t, u):
        z = 2.0 * self.gamma * t
        p1 = math.expm1(z) / z if z else 1.0
        L = torch.log1p(2.0 * t * p1 * self.kappa * (u.real ** 2 + u.imag ** 2))
        return torch.exp(t * self.gamma - (self.kappa + 1j * self.zeta) / (2.0 * self.kappa) * L) * u

    def integrate(self, scheme, tau, steps, u):
        A = self.apply
        prev = u
        for n in range(steps):
            t = n * tau
            if scheme == "lie" or (scheme == "lbdf2" and n == 0):
                prev, u = u, A("inv", 0, tau, u + tau * self.g(t, u))
            elif scheme == "lbdf2":
                rhs = (4.0 * u - prev) / 3.0 + (2.0 * tau / 3.0) * self.g(t + tau, 2.0 * u - prev)
                prev, u = u, A("inv", 0, 2.0 * tau / 3.0, rhs)
            elif scheme == "lawson_euler":
                u = A("exp", 0, tau, u + tau * self.g(t, u))
            elif scheme == "lawson_rk2":
                k1 = self.g(t, u)
                v = A("exp", 0, tau, u + tau * k1)
                u = A("exp", 0, tau, u + 0.5 * tau * k1) + 0.5 * tau * self.g(t + tau, v)
            elif scheme == "strang":
                u = self.flow(tau / 2, A("exp", 0, tau, self.flow(tau / 2, u)))
            else:
                Ku = self.bwd(self.Lam * self.fwd(u))
                gn = self.g(t, u)
                fn = Ku + gn
                if scheme == "etd2rk":
                    a = u + tau * A("phi", 1, tau, fn)
                    u = a + tau * A("phi", 2, tau, self.g(t + tau, a) - gn)
                else:
                    h = tau / 2
                    d2 = self.g(t + h, u + h * A("phi", 1, h, fn)) - gn
                    d3 = self.g(t + h, u + tau * (0.5 * A("phi", 1, h, fn) + A("phi", 2, h, d2))) - gn
                    d4 = self.g(t + tau, u + tau * (A("phi", 1, tau, fn) + 2.0 * A("phi", 2, tau, d3))) - gn
                    u = u + tau * (A("phi", 1, tau, fn) + A("phi", 2, tau, 2.0 * d2 + 2.0 * d3 - d4)
                                   + A("phi", 3, tau, 4.0 * (d4 - d2 - d3)))
        return u


def exact(case, seed):
    dev = _device()
    u0 = _u0(case, seed, dev)
    if case["kind"] == "batch":
        out = []
        for sp, u in zip(_specs(case), u0):
            e = _Exact(sp["ns"], sp["boxes"], sp["alphas"], sp["nu"], sp["eta"], sp["gamma"], sp["kappa"], sp["zeta"], dev)
            out.append(e.integrate(case["scheme"], case["tau"], case["steps"], u.to(torch.complex128)))
        return out
    ns, box, d = _ns(case), case["box"], len(_ns(case))
    sig, S = _source(ns, box, case.get("source", 0), dev)
    S = [x.to(_dtype(case)).to(torch.complex128) for x in S]
    u = u0.to(torch.complex128)
    if case["kind"] == "adjoint":
        pars = torch.tensor(COEFFS, dtype=torch.float64, device=dev, requires_grad=True)
        target = _target(case, u0).to(torch.complex128)
        u.requires_grad_(True)
        e = _Exact(ns, [(-box, box)] * d, ALPHAS[d], *pars.unbind(), dev)
        uT = e.integrate("lawson_rk2", case["tau"], case["steps"], u)
        diff = uT - target
        loss = 0.5 * (diff.real ** 2 + diff.imag ** 2).sum()
        gu, gp = torch.autograd.grad(loss, [u, pars])
        return dict(loss=float(loss.detach()), grad_u0=gu, grad_params=gp.cpu())
    e = _Exact(ns, [(-box, box)] * d, ALPHAS[d], *COEFFS, dev, sig, S)
    if case["kind"] == "apply":
        return e.apply(case["func"], case["k"], case["theta"], u)
    return e.integrate(case["scheme"], case["tau"], case["steps"], u)
