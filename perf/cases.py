"""What a program that uses this library has it do: the calls that are timed and compared.

Every case goes through the public entry points (``ks_residual``, the autograd ``cost``,
``ks_descend`` and the chaotic run ``ks_dns``) with device buffers, as the tests, the benchmark
and the orbit search do.  The loops are seeded spectral loops of the repository's workloads
(normal coefficients with exponential decay, zero mean, grid rms 1), drawn here from the seed
alone; the trajectories start from the small seeded perturbation of a chaotic run.

Mixed handles run the double and float steps of the cases below; their outputs are double arrays
that hold float-rounded values until the double finish, which takes seconds, so no case of their
own: the two precisions are listed side by side instead.

A float handle returns its period, cost and sqrt(J) in double arrays that hold values of float
accuracy, so a float program keeps them as floats: ``run`` hands them back in the descent's type.
"""
import math

import numpy as np
import torch

from paper_2007_06427_gb300 import ks_loop as K
from paper_2007_06427_gb300.autograd import cost

DEV = "cuda"


def listed():
    return [
        # the smallest call: r and J of one 32 x 32 loop, a few launches from end to end
        dict(name="residual_32x32_f64", kind="residual", L=22.0, nx=32, ns="32", B=1, T_lo=40.0,
             T_hi=40.0, dx=2.0, ds=2.0, f32=False, xi=False),
        # the plain method: one small loop under explicit steps within the stiffness limit
        dict(name="explicit_32x32_f64", kind="descend", L=22.0, nx=32, ns="32", B=1, T_lo=40.0,
             T_hi=40.0, dx=2.0, ds=2.0, f32=False, xi=False, imex=False, dtau=1e-4, steps=500),
        # the benchmark's loop, in double and in float: one loop, bound by latency
        dict(name="descend_64x128_f64", kind="descend", L=22.0, nx=64, ns="128", B=1, T_lo=20.0,
             T_hi=80.0, dx=2.0, ds=2.0, f32=False, xi=False, imex=True, dtau=0.15, steps=200),
        dict(name="descend_64x128_f32", kind="descend", L=22.0, nx=64, ns="128", B=1, T_lo=20.0,
             T_hi=80.0, dx=2.0, ds=2.0, f32=True, xi=False, imex=True, dtau=0.15, steps=400),
        # differentiation: J(u, T) and its gradient for a batch of 16, forward and backward
        dict(name="grad16_64x64_f64", kind="grad", L=22.0, nx=64, ns="64", B=16, T_lo=20.0,
             T_hi=80.0, dx=2.0, ds=2.0, f32=False, xi=False),
        dict(name="grad16_64x64_f32", kind="grad", L=22.0, nx=64, ns="64", B=16, T_lo=20.0,
             T_hi=80.0, dx=2.0, ds=2.0, f32=True, xi=False),
        # batching: 256 loops of uneven length, the bulk of a search in double and in float
        dict(name="ragged256_f64", kind="descend", L=22.0, nx=64, ns="32,64,128,256", B=256,
             T_lo=10.0, T_hi=100.0, dx=2.0, ds=2.0, f32=False, xi=False, imex=True, dtau=0.15,
             steps=40),
        dict(name="ragged256_f32", kind="descend", L=22.0, nx=64, ns="32,64,128,256", B=256,
             T_lo=10.0, T_hi=100.0, dx=2.0, ds=2.0, f32=True, xi=False, imex=True, dtau=0.15,
             steps=120),
        # the large domain: eight 256 x 1024 loops, in double and in float
        dict(name="large8_256x1024_f64", kind="descend", L=100.0, nx=256, ns="1024", B=8,
             T_lo=120.0, T_hi=120.0, dx=8.0, ds=8.0, f32=False, xi=False, imex=True, dtau=0.15,
             steps=20),
        dict(name="large8_256x1024_f32", kind="descend", L=100.0, nx=256, ns="1024", B=8,
             T_lo=120.0, T_hi=120.0, dx=8.0, ds=8.0, f32=True, xi=False, imex=True, dtau=0.15,
             steps=60),
        # the paper's setting: centre-symmetric loops at L = 39, a batch of an orbit search
        dict(name="orbits16_xi_64x64_f64", kind="descend", L=39.0, nx=64, ns="64", B=16,
             T_lo=20.0, T_hi=120.0, dx=2.0, ds=2.0, f32=False, xi=True, imex=True, dtau=0.15,
             steps=100),
        # the run behind the initial loops: centre-symmetric chaotic trajectories
        dict(name="dns64_L39_64", kind="dns", L=39.0, nx=64, B=64, dt=0.25, steps=240, save=2,
             xi=True),
    ]


# domain lengths that a grid of nx points resolves
_L = {32: (16.0, 24.0), 64: (20.0, 40.0), 128: (30.0, 60.0), 256: (60.0, 110.0)}
# gridpoint-steps of the largest listed cases, by element type
_MOST = {False: 8 * 256 * 1024 * 20, True: 8 * 256 * 1024 * 60}


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["residual", "grad", "descend", "descend", "descend", "descend", "dns"])
    if kind == "dns":
        nx = rng.choice([32, 64, 64, 128])
        return dict(kind="dns", L=round(rng.uniform(*_L[nx]), 3), nx=nx,
                    B=int(_log(rng, 1, 300)), dt=rng.choice([0.2, 0.25]),
                    steps=rng.randrange(41, 240), save=rng.choice([1, 2, 3, 5]),
                    xi=rng.random() < 0.5)
    f32 = rng.random() < 0.4
    nx = rng.choice([32, 64, 64, 64, 128, 256])
    lens = rng.choice(["32", "64", "128", "256", "16,64", "32,64,128", "32,64,128,256"]
                      + (["512", "1024"] if nx >= 128 else []))
    longest = max(int(v) for v in lens.split(","))
    mean = sum(int(v) for v in lens.split(",")) / len(lens.split(","))
    B = int(_log(rng, 1, 300))
    B = max(1, min(B, int(_MOST[f32] / (5 * nx * mean)), 2048 * 1024 // (nx * longest)))
    d = 2.0 if longest < 512 else 8.0
    c = dict(kind=kind, L=round(rng.uniform(*_L[nx]), 3), nx=nx, ns=lens, B=B, T_lo=20.0,
             T_hi=100.0, dx=nx / 32.0 if nx > 64 else 2.0, ds=d, f32=f32,
             xi=rng.random() < 0.25)
    if kind == "descend":
        most = max(2, int(_MOST[f32] / (B * nx * mean)))
        c["imex"] = rng.random() < 0.9
        q = 2 * math.pi * (nx // 3) / c["L"]     # explicit steps stay within the stiffness limit
        c["dtau"] = round(rng.uniform(0.05, 0.2), 3) if c["imex"] else 0.3 / (q * q * (q * q - 1)) ** 2
        c["steps"] = int(_log(rng, 2, max(3, min(301, most))))
    return c


# ---- inputs ------------------------------------------------------------------------------

def _loops(case, seed):
    """(lengths, fields, periods) of the batch: float64 fields u[n, m] on the host."""
    nx, kx = case["nx"], case["nx"] // 3
    lens = [int(v) for v in case["ns"].split(",")]
    # the lengths belong to the case (a handle is made for them), the fields to the seed
    ns = [int(v) for v in np.random.default_rng(case["B"]).choice(lens, case["B"])]
    rng = np.random.default_rng(seed)
    T = rng.uniform(case["T_lo"], case["T_hi"], case["B"])
    us = []
    j = np.arange(kx + 1)
    for n in ns:
        ks = n // 3
        k = np.arange(-ks, ks + 1)
        c = rng.standard_normal((kx + 1, 2 * ks + 1)) + 1j * rng.standard_normal((kx + 1, 2 * ks + 1))
        c *= np.exp(-j / case["dx"])[:, None] * np.exp(-np.abs(k) / case["ds"])[None, :]
        c[0] = 0.0
        if case["xi"]:
            c = 0.5 * (c - np.conj(c[:, ::-1]))
        half = np.zeros((n, nx // 2 + 1), dtype=complex)
        half[k % n, : kx + 1] = c.T
        u = np.fft.irfft2(half, s=(n, nx))
        us.append(u / np.sqrt(np.mean(u * u)))
    return ns, us, T


def _starts(case, seed):
    """The perturbations that chaotic runs start from, [B, nx]."""
    rng = np.random.default_rng(seed)
    x = 2 * np.pi * np.arange(case["nx"]) / case["nx"]
    a = rng.standard_normal((case["B"], 2))
    return (a[:, :1] * np.cos(x) + a[:, 1:] * np.sin(2 * x)
            + 0.3 * rng.standard_normal((case["B"], case["nx"])))


def prepare(case, seed):
    if case["kind"] == "dns":
        return dict(case, u0=torch.from_numpy(_starts(case, seed)).to(DEV))
    ns, us, T = _loops(case, seed)
    dt = torch.float32 if case["f32"] else torch.float64
    u = torch.from_numpy(np.concatenate([v.ravel() for v in us])).to(DEV).to(dt)
    h = K.KSLoop(case["L"], case["nx"], ns, K.KS_FP32 if case["f32"] else K.KS_FP64,
                 K.KS_IMEX if case.get("imex", True) else K.KS_EXPLICIT, case.get("dtau", 0.15))
    if case["xi"]:
        K.ks_set_option(h.handle, "symmetry", 1)
    return dict(case, loop=h, u=u, T=torch.from_numpy(T).to(DEV), dtype=dt)


# ---- one pass ----------------------------------------------------------------------------

def run(s):
    return {"residual": _residual, "grad": _grad, "descend": _descend, "dns": _dns}[s["kind"]](s)


def _residual(s):
    r = torch.empty_like(s["u"])
    J = torch.empty_like(s["T"])
    K.ks_residual(s["loop"].handle, s["u"], s["T"], r, J, torch.cuda.current_stream())
    return {"r": r, "J": J.to(s["dtype"])}


def _grad(s):
    u = s["u"].detach().requires_grad_()
    T = s["T"].detach().requires_grad_()
    J = cost(u, T, s["loop"])
    J.sum().backward()
    return {"J": J.detach().to(s["dtype"]), "u_grad": u.grad, "T_grad": T.grad.to(s["dtype"])}


def _descend(s):
    u, T = s["u"].clone(), s["T"].clone()
    B = s["B"]
    steps = torch.empty(B, dtype=torch.int64, device=DEV)
    sq = torch.empty(B, dtype=torch.float64, device=DEV)
    status = torch.empty(B, dtype=torch.int32, device=DEV)
    K.ks_descend(s["loop"].handle, u, T, s["steps"], 1e-10, steps, sq, status,
                 torch.cuda.current_stream())
    return {"u": u, "T": T.to(s["dtype"]), "steps": steps, "sqrtJ": sq.to(s["dtype"]),
            "status": status}


def _dns(s):
    nsave = s["steps"] // s["save"] + 1
    us = torch.empty(s["B"], nsave, s["nx"], dtype=torch.float64, device=DEV)
    norms = torch.empty(s["B"], nsave, dtype=torch.float64, device=DEV)
    end = torch.empty(s["B"], s["nx"], dtype=torch.float64, device=DEV)
    K.ks_dns(s["L"], s["nx"], s["B"], s["dt"], s["steps"], s["save"], s["xi"], s["u0"], us, norms,
             end, torch.cuda.current_stream())
    return {"u": us, "norms": norms, "end": end}


# ---- what a pass cannot do without -------------------------------------------------------

def work(case):
    nx, B = case["nx"], case["B"]
    if case["kind"] == "dns":
        nsave = case["steps"] // case["save"] + 1
        # four evaluations a step: one inverse and one forward real transform and the product,
        # then the stages of the scheme on the half spectrum
        step = 4 * (2 * 2.5 * nx * math.log2(nx) + 10 * nx) + 30 * (nx // 3 + 1)
        return {"bytes": 8.0 * B * (nx * (2 + nsave) + nsave), "flops": B * case["steps"] * step}
    lens = [int(v) for v in case["ns"].split(",")]
    e = 4 if case["f32"] else 8
    pts = B * nx * sum(lens) / len(lens)                       # mean over the drawn lengths
    tr = B * sum(2.5 * nx * n * math.log2(nx * n) for n in lens) / len(lens)  # one real transform
    if case["kind"] == "residual":   # analysis, two inverse, one forward, synthesis
        return {"bytes": 2 * e * pts + 16 * B, "flops": 5 * tr + 20 * pts}
    if case["kind"] == "grad":       # the same with the adjoint's two transforms
        return {"bytes": 2 * e * pts + 24 * B, "flops": 7 * tr + 40 * pts}
    steps = case["steps"]            # five real transforms and the pointwise terms per step
    return {"bytes": 2 * e * pts + 36 * B, "flops": steps * (5 * tr + 40 * pts)}


# ---- the same in 64 bits -----------------------------------------------------------------

class _Group:
    """Loops of one length, as a batch [b, n, m] of torch arrays in 64 bits."""

    def __init__(self, case, u, T):
        nx, n, L = case["nx"], u.shape[1], case["L"]
        self.xi, self.L, self.n, self.nx = case["xi"], L, n, nx
        q = 2 * math.pi * torch.arange(nx // 2 + 1, dtype=torch.float64, device=DEV) / L
        k = torch.fft.fftfreq(n, 1.0 / n, dtype=torch.float64, device=DEV)
        self.q, self.om = q[None, None, :], 2 * math.pi * k[None, :, None]
        self.keep = ((torch.arange(nx // 2 + 1, device=DEV)[None, None, :] <= nx // 3)
                     & (k.abs()[None, :, None] <= n // 3))
        self.w = torch.full_like(self.q, 2.0)
        self.w[..., 0] = 1.0
        self.T = T[:, None, None].clone()
        self.uh = self.project(self.band(u))

    def band(self, f):
        return torch.fft.rfft2(f, norm="forward") * self.keep

    def grid(self, fh):
        return torch.fft.irfft2(fh, s=(self.n, self.nx), norm="forward")

    def project(self, fh):
        if not self.xi:
            return fh
        mirror = torch.roll(torch.flip(fh, dims=(1,)), 1, dims=1)       # k -> -k
        fh = 0.5 * (fh - mirror.conj())
        fh[..., 0] = 0
        return fh

    def residual(self):
        q, om = self.q, self.om
        self.u = self.grid(self.uh)
        p = self.band(self.u * self.grid(1j * q * self.uh))
        self.rh = (-1j * om / self.T + q**2 - q**4) * self.uh - p
        self.J = self.L * (self.w * self.rh.abs() ** 2).sum((1, 2))
        s = (self.w * om * (self.uh.conj() * self.rh).imag).sum((1, 2))
        self.L2 = self.L * s / self.T[:, 0, 0] ** 2

    def gradient(self):
        q, om = self.q, self.om
        self.residual()
        a = self.band(self.u * self.grid(1j * q * self.rh))
        return self.project((1j * om / self.T + q**2 - q**4) * self.rh + a)

    def step(self, dtau, imex):
        G = self.gradient()
        if imex:
            lam = -(self.om / self.T) ** 2 - self.q**4 * (self.q**2 - 1) ** 2
            G = G / (1 - dtau * lam)
        self.uh = self.uh - dtau * G
        self.T = self.T - dtau * self.L2[:, None, None]


def _exact_dns(case, seed):
    L, nx, dt, B = case["L"], case["nx"], case["dt"], case["B"]
    kx = nx // 3
    q = 2 * np.pi * np.arange(nx // 2 + 1) / L
    z = (dt * (q**2 - q**4)).astype(np.longdouble)
    # the weights of the scheme as means over a circle around z (Kassam & Trefethen), in more
    # than 64 bits where the host has them
    th = np.pi * (np.arange(64).astype(np.longdouble) + np.longdouble(0.5)) / 32
    r = z[:, None] + np.cos(th) + 1j * np.sin(th)
    e = np.exp(r)
    f = lambda x: torch.from_numpy(x.mean(1).real.astype(np.float64) * dt).to(DEV)  # noqa: E731
    Q = f((np.exp(r / 2) - 1) / r)
    f1 = f((-4 - r + e * (4 - 3 * r + r**2)) / r**3)
    f2 = f((2 + r + e * (r - 2)) / r**3)
    f3 = f((-4 - 3 * r - r**2 + e * (4 - r)) / r**3)
    E = torch.from_numpy(np.exp(z).astype(np.float64)).to(DEV)
    E2 = torch.from_numpy(np.exp(z / 2).astype(np.float64)).to(DEV)
    qd = torch.from_numpy(q).to(DEV)
    keep = (torch.arange(nx // 2 + 1, device=DEV) <= kx).to(torch.float64)

    def sym(v):
        return torch.complex(torch.zeros_like(v.real), v.imag) if case["xi"] else v

    def grid(v):
        return torch.fft.irfft(v, n=nx)

    def nonlin(v):
        return -0.5j * qd * keep * torch.fft.rfft(grid(v) ** 2)

    v = sym(keep * torch.fft.rfft(torch.from_numpy(_starts(case, seed)).to(DEV)))
    saved = []
    for i in range(case["steps"] + 1):
        if i % case["save"] == 0:
            saved.append(grid(v))
        if i == case["steps"]:
            break
        Nv = nonlin(v)
        a = E2 * v + Q * Nv
        Na = nonlin(a)
        b = E2 * v + Q * Na
        Nb = nonlin(b)
        c = E2 * a + Q * (2 * Nb - Nv)
        v = sym(E * v + f1 * Nv + 2 * f2 * (Na + Nb) + f3 * nonlin(c))
    us = torch.stack(saved, dim=1)
    return {"u": us, "norms": (us.square().mean(-1) * L).sqrt(), "end": grid(v)}


def exact(case, seed):
    if case["kind"] == "dns":
        return _exact_dns(case, seed)
    ns, us, T = _loops(case, seed)
    if case["f32"]:  # a float program hands the field over in float
        us = [u.astype(np.float32).astype(np.float64) for u in us]
    B = case["B"]
    fields = [None] * B
    J = torch.zeros(B, dtype=torch.float64, device=DEV)
    dT, Tn = torch.zeros_like(J), torch.zeros_like(J)
    for n in sorted(set(ns)):
        at = [b for b in range(B) if ns[b] == n]
        g = _Group(case, torch.from_numpy(np.stack([us[b] for b in at])).to(DEV),
                   torch.from_numpy(T[at]).to(DEV))
        if case["kind"] == "residual":
            g.residual()
            out = g.grid(g.rh)
        elif case["kind"] == "grad":
            out = g.grid(g.gradient()) * (2 * case["L"] / (case["nx"] * n))
        else:
            for _ in range(case["steps"]):
                g.step(case["dtau"], case["imex"])
            g.residual()
            out = g.grid(g.uh)
        for i, b in enumerate(at):
            fields[b] = out[i].reshape(-1)
            J[b], dT[b], Tn[b] = g.J[i], 2 * g.L2[i], g.T[i, 0, 0]
    u = torch.cat(fields)
    if case["kind"] == "residual":
        return {"r": u, "J": J}
    if case["kind"] == "grad":
        return {"J": J, "u_grad": u, "T_grad": dT}
    return {"u": u, "T": Tn, "steps": None, "sqrtJ": J.sqrt(), "status": None}
