"""What is timed: the calls that users of this framework make, through its public entry points, over the
range of grids, batches, windows and options that it serves.

Grids are the powers of two from 16 to 1024 that the library supports; window lengths, batches, probe
lattices, observation intervals, kernels and viscosities take any value, odd ones among them.
"""
from __future__ import annotations

import math

import torch

from paper_2602_14016_gb300 import api, autograd

# the kernel sweep |k|^(-2s), exp(-a|k|) of the 256^2 workload
SWEEP = [("frac", 0.0), ("frac", 0.5), ("frac", 1.0), ("frac", 1.5), ("exp_abs", 0.1), ("exp_abs", 0.3),
         ("exp_abs", 1.0)]

BASE = dict(kind="cost_grad", n=64, batch=1, nsteps=10, dt=5e-3, nu=1e-3, forced=False, px=8, every=5, t0=False,
            kernel="exp_abs", param=0.5, ckpt=0, graphs=True, tune=True, iters=0)


def _case(**kw):
    return {**BASE, **kw}


def listed():
    return [
        # the control map and its inverse on their own: what a program that proposes or inspects controls calls
        # between evaluations; a handful of launches
        _case(name="maps256x7", kind="maps", n=256, batch=7, nsteps=1, every=1, px=16, dt=2e-3, kernel="sweep",
              graphs=False, tune=False),
        # the smallest evaluation: a 16^2 window of a few steps, launched directly (no graph, no tuning)
        _case(name="cost_grad16", n=16, nsteps=6, dt=1e-2, px=8, every=3, t0=True, kernel="frac", param=1.0,
              graphs=False, tune=False),
        # the plain method's window: 64^2, 200 steps, one member, replayed as a graph
        _case(name="cost_grad64", n=64, nsteps=200, dt=5e-3, px=8, every=10),
        # one member at 128^2, heat kernel, denser probes
        _case(name="cost_grad128", n=128, nsteps=100, dt=4e-3, nu=5e-4, px=16, every=10, kernel="exp_sq", param=0.7),
        # the headline workload on a shorter window: forced 256^2, the seven kernels as one batch
        _case(name="sweep256x7", n=256, batch=7, nsteps=200, dt=2e-3, nu=1e-2, forced=True, px=16, every=20,
              kernel="sweep"),
        # one 256^2 member with checkpoints (a long window that does not fit as full storage)
        _case(name="ckpt256", n=256, nsteps=60, dt=2e-3, nu=1e-2, forced=True, px=16, every=20, kernel="frac",
              param=0.5, ckpt=25),
        # the largest grid
        _case(name="cost_grad1024", n=1024, nsteps=8, dt=5e-4, px=32, every=4, kernel="exp_abs", param=0.2),
        # forward only, no stored trajectory: spin-up and data generation for a batch, launched directly
        _case(name="forward256x5", kind="forward", n=256, batch=5, nsteps=50, dt=2e-3, nu=1e-2, forced=True, px=16,
              every=10, kernel="identity", param=0.0, graphs=False, tune=False),
        # the differentiable 512^2 window: forward and backward through torch.autograd
        _case(name="autograd512", kind="autograd", n=512, nsteps=20, dt=1e-3, nu=5e-3, forced=True, px=32, every=10,
              kernel="frac", param=0.5, graphs=False),
        # adjoint statistics of an ensemble: shell spectra of the adjoint along the backward time
        _case(name="spectra256x16", kind="spectra", n=256, batch=16, nsteps=40, dt=2e-3, nu=1e-3, px=1, every=10,
              kernel="identity", param=0.0, ckpt=20),
        # a serving pool: jobs with windows of their own share the launches of one evaluation
        _case(name="ragged64x13", kind="ragged", n=64, batch=13, nsteps=60, dt=5e-3, forced=True, px=16, every=5),
        # a whole assimilation, short: L-BFGS with its line search around the evaluations
        _case(name="assimilate64x3", kind="assimilate", n=64, batch=3, nsteps=40, dt=5e-3, px=8, every=10, iters=3),
    ]


def _cost(c):
    f = {"maps": 1.0 / 32, "forward": 0.5, "assimilate": 1.5 * c["iters"] + 1}.get(c["kind"], 1.0)
    return f * c["batch"] * c["n"] ** 2 * math.log2(c["n"]) * c["nsteps"] * (1.5 if c["ckpt"] else 1.0)


def draw(rng):
    most = max(_cost(c) for c in listed())
    while True:
        kind = rng.choice(["cost_grad"] * 5 + ["maps", "forward", "autograd", "spectra", "ragged"])
        n = rng.choice([16, 32, 64, 64, 128, 128, 256, 256, 512, 1024])
        batch = 1 if kind == "autograd" else round(math.exp(rng.uniform(0, math.log(24))))
        every = rng.randint(1, 12)
        nsteps = 1 if kind == "maps" else every * rng.randint(1, max(1, round(math.exp(rng.uniform(0, math.log(200)))) // every))
        kernel, param = rng.choice([("identity", 0.0), ("sweep", 0.0), ("frac", rng.uniform(0.2, 1.5)),
                                    ("exp_abs", rng.uniform(0.05, 0.6)), ("exp_sq", rng.uniform(0.1, 0.8))])
        if kind == "spectra":
            kernel, param = "identity", 0.0
        c = _case(kind=kind, n=n, batch=batch, nsteps=nsteps, every=1 if kind == "maps" else every,
                  dt=0.4 / n * rng.uniform(0.3, 1.0), nu=math.exp(rng.uniform(math.log(5e-4), math.log(1e-2))),
                  forced=rng.random() < 0.5, px=2 ** rng.randint(0, min(6, int(math.log2(n)))), t0=rng.random() < 0.3,
                  kernel=kernel, param=param, graphs=kind not in ("maps", "forward", "autograd") and rng.random() < 0.8,
                  tune=kind not in ("maps", "forward") and rng.random() < 0.5,
                  ckpt=rng.randint(1, max(1, nsteps - 1)) if kind in ("cost_grad", "spectra", "autograd") and
                  nsteps > 2 and rng.random() < 0.25 else 0)
        if _cost(c) <= 0.8 * most and _cost(c) >= 1e4:
            return c


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _wave(n, dev):
    kx = torch.arange(n // 2 + 1, device=dev, dtype=torch.float64)[None, :]
    ky = torch.fft.fftfreq(n, 1.0 / n, device=dev, dtype=torch.float64)[:, None]
    K = (n - 1) // 3
    keep = ((kx.abs() <= K) & (ky.abs() <= K)).double()
    k2 = kx * kx + ky * ky
    ik2 = torch.where(k2 > 0, 1.0 / torch.where(k2 > 0, k2, 1.0), 0.0)
    return kx, ky, k2, ik2, keep


def _kernels(c):
    if c["kernel"] == "sweep":
        return [SWEEP[b % len(SWEEP)] for b in range(c["batch"])]
    return [(c["kernel"], c["param"])] * c["batch"]


def _multiplier(c, nus, dev):
    """|k| W^(1/2) of every member on the retained set."""
    _, _, k2, _, keep = _wave(c["n"], dev)
    k = k2.sqrt()
    ks = torch.where(k > 0, k, 1.0)
    out = []
    for (kind, a), nu in zip(_kernels(c), nus):
        w = {"identity": lambda: torch.ones_like(k), "exp_abs": lambda: torch.exp(-a * k),
             "frac": lambda: ks ** (-2.0 * a), "exp_sq": lambda: torch.exp(-nu * a * k2)}[kind]()
        out.append(k * w.sqrt() * keep)
    return torch.stack(out)


def _vorticity(c, gen, dev):
    """Random-phase vorticity, E(k) ~ k^4 exp(-2 (k/4)^2), unit energy: half spectra [batch, n, n/2+1]."""
    n = c["n"]
    _, _, k2, ik2, keep = _wave(n, dev)
    k = k2.sqrt()
    h = torch.fft.rfft2(torch.randn((c["batch"], n, n), generator=gen, device=dev, dtype=torch.float64))
    h = h / h.abs().clamp_min(1e-300) * (k * k ** 4 * torch.exp(-2.0 * (k / 4.0) ** 2)).sqrt() * keep
    wt = torch.full((n // 2 + 1,), 2.0, device=dev, dtype=torch.float64)
    wt[0] = 1.0
    e = 0.5 / n ** 4 * (wt * h.abs() ** 2 * ik2).sum(dim=(1, 2), keepdim=True)
    return h / e.sqrt()


def _windows(c):
    """(nsteps, px, nu, forced) of every member: the context's, or a spread of shorter ones in a ragged pool."""
    if c["kind"] != "ragged":
        return [(c["nsteps"], c["px"], c["nu"], c["forced"])] * c["batch"]
    most = c["nsteps"] // c["every"]
    return [(c["every"] * (most - (b * 5) % most), max(1, c["px"] >> (b % 3)), c["nu"] * (1 + 0.25 * (b % 4)),
             c["forced"] and b % 2 == 0) for b in range(c["batch"])]


def _velocity(w, n):
    kx, ky, _, ik2, _ = _wave(n, w.device)
    return torch.fft.irfft2(1j * ky * ik2 * w, s=(n, n)), torch.fft.irfft2(-1j * kx * ik2 * w, s=(n, n))


def _inputs(c, seed):
    """Control of a first guess, probe data (a truth's velocities with 1 % noise at every time) and a terminal field."""
    dev = torch.device("cuda")
    gen = torch.Generator(device=dev)
    gen.manual_seed(seed)
    n = c["n"]
    u, v = _velocity(_vorticity(c, gen, dev), n)
    data = []
    for b, (steps, px, _, _) in enumerate(_windows(c)):
        nt = steps // c["every"] + (1 if c["t0"] else 0)
        st = n // px
        o = torch.stack([u[b, ::st, ::st].reshape(-1), v[b, ::st, ::st].reshape(-1)], dim=-1)
        noise = torch.randn((nt, px * px, 2), generator=gen, device=dev, dtype=torch.float64)
        data.append(o + 0.01 * o.square().mean().sqrt() * noise)
    w0 = _vorticity(c, gen, dev)
    m = _multiplier(c, [x[2] for x in _windows(c)], dev)
    s = torch.fft.irfft2(torch.where(m > 0, w0 / torch.where(m > 0, m, 1.0), 0.0), s=(n, n)).contiguous()
    lam = torch.fft.rfft2(torch.randn((c["batch"], n, n), generator=gen, device=dev, dtype=torch.float64))
    lam = lam * _wave(n, dev)[4]
    f = torch.fft.irfft2(lam, s=(n, n))
    lam = (lam / f.square().sum(dim=(1, 2), keepdim=True).sqrt()).contiguous()
    return s, data, w0.contiguous(), lam


def prepare(case, seed):
    c = case
    s, data, w0, lam = _inputs(c, seed)
    ctx = api.Context(api.Config(
        n=c["n"], nsteps=c["nsteps"], dt=c["dt"], nu=c["nu"], forcing="kolmogorov" if c["forced"] else "none",
        nf=4, px=c["px"], every=c["every"], include_t0=c["t0"],
        kernels=[api.KernelSpec(k, a) for k, a in _kernels(c)], ckpt_every=c["ckpt"],
        store=c["kind"] not in ("forward", "maps")))
    if c["tune"]:
        ctx.autotune(4)
    if c["graphs"]:
        ctx.set_graphs(True)
    st = {"case": c, "ctx": ctx, "s": s, "w0": w0, "lam": lam}
    if c["kind"] == "ragged":
        for b, (steps, px, nu, forced) in enumerate(_windows(c)):
            ctx.set_member(b, steps, px=px, nu=nu, forcing=forced, kernel=api.KernelSpec(*_kernels(c)[b]), m=data[b])
    elif c["kind"] in ("cost_grad", "assimilate"):
        ctx.set_observations(torch.stack(data))
    elif c["kind"] == "autograd":
        st["m"] = torch.stack(data)
    return st


def run(state):
    c, ctx, s = state["case"], state["ctx"], state["s"]
    if c["kind"] == "maps":
        return {"w": ctx.omega_from_control(s), "s": ctx.control_from_omega(state["w0"])}
    if c["kind"] == "forward":
        w, obs = ctx.forward(s)
        return {"w": w, "obs": obs}
    if c["kind"] == "spectra":
        member, mean = ctx.adjoint_spectra(s, state["lam"], c["every"])
        lam0, filtered = ctx.last_adjoint()
        return {"member": member, "mean": mean, "lam0": lam0, "filtered": filtered}
    if c["kind"] == "autograd":
        x = s.detach().clone().requires_grad_(True)
        obs, w = autograd.solve(x, ctx)
        loss = autograd.misfit(obs, state["m"]).sum()
        (g,) = torch.autograd.grad(loss, x)
        return {"obs": obs.detach(), "w": w.detach(), "loss": loss.detach(), "grad": g}
    if c["kind"] == "assimilate":
        x = s.clone()
        res = ctx.assimilate(x, c["iters"])
        return {"s": x, "J": res.J_hist, "iters": res.iters}
    J, g = ctx.cost_grad(s)
    return {"J": J, "grad": g}


def work(case):
    """Inputs read once, outputs written once; the flops of the transforms (a real 2D transform of n^2 points on the
    2/3-rule band: 2.5 n log2 n for each row and 5 n log2 n for each kept column) and of the arithmetic between
    them.  A stage: two inverse and two forward transforms each way."""
    c = case
    n, B = c["n"], c["batch"]
    K = (n - 1) // 3
    lg = math.log2(n)
    t2d = n * 2.5 * n * lg + (K + 1) * 5.0 * n * lg
    fwd = 4 * (4 * t2d + 3.0 * n * n + 26.0 * (K + 1) * (2 * K + 1))
    adj = 4 * (4 * t2d + 6.0 * n * n + 32.0 * (K + 1) * (2 * K + 1))
    field, spec = 8.0 * n * n, 16.0 * n * (n // 2 + 1)
    steps = [w[0] for w in _windows(c)]
    obs = sum(16.0 * w[1] ** 2 * (w[0] // c["every"] + (1 if c["t0"] else 0)) for w in _windows(c))
    if c["kind"] == "maps":
        return {"bytes": B * 2 * (field + spec), "flops": B * 2 * t2d}
    if c["kind"] == "forward":
        return {"bytes": B * (field + spec) + obs, "flops": sum(steps) * fwd + B * t2d}
    flops = sum(steps) * (fwd + adj) + B * 2 * t2d
    if c["kind"] == "spectra":
        shells = (c["nsteps"] // c["every"] + 1) * (int(math.sqrt(2.0) * K) + 1)
        return {"bytes": B * 2 * (field + spec) + 8.0 * (B + 1) * shells, "flops": flops}
    if c["kind"] == "autograd":
        return {"bytes": B * (2 * field + spec) + 2 * obs, "flops": flops}
    if c["kind"] == "assimilate":
        return {"bytes": B * 2 * field + obs, "flops": flops * (c["iters"] + 1)}
    return {"bytes": B * 2 * field + obs, "flops": flops}


# ---------------------------------------------------------------------------
# the same in 64 bits, by torch alone
# ---------------------------------------------------------------------------

class _Plain:
    """The vorticity equation with RK4 and the 2/3 rule on half spectra, advective form."""

    def __init__(self, c, dev):
        self.n, self.dt = c["n"], c["dt"]
        self.kx, self.ky, self.k2, self.ik2, self.keep = _wave(c["n"], dev)
        wins = _windows(c)
        self.nu = torch.tensor([w[2] for w in wins], device=dev, dtype=torch.float64)[:, None, None]
        self.f = torch.zeros((len(wins), c["n"], c["n"] // 2 + 1), device=dev, dtype=torch.complex128)
        for b, w in enumerate(wins):
            if w[3]:
                self.f[b, 4, 0] = self.f[b, -4, 0] = -4.0 * c["n"] ** 2 / 2.0

    def inv(self, h):
        return torch.fft.irfft2(h, s=(self.n, self.n))

    def rhs(self, w):
        u, v = self.inv(1j * self.ky * self.ik2 * w), self.inv(-1j * self.kx * self.ik2 * w)
        a = torch.fft.rfft2(u * self.inv(1j * self.kx * w) + v * self.inv(1j * self.ky * w))
        return self.f - self.keep * a - self.nu * self.k2 * w

    def step(self, w):
        h = self.dt
        k1 = self.rhs(w)
        k2 = self.rhs(w + 0.5 * h * k1)
        k3 = self.rhs(w + 0.5 * h * k2)
        k4 = self.rhs(w + h * k3)
        return w + h / 6.0 * (k1 + 2 * k2 + 2 * k3 + k4)


def exact(case, seed):
    c = case
    if c["kind"] == "assimilate" or c["nsteps"] > 1000:
        return None
    dev = torch.device("cuda")
    n = c["n"]
    s, data, w0, lamT = _inputs(c, seed)
    wins = _windows(c)
    mult = _multiplier(c, [w[2] for w in wins], dev)
    if c["kind"] == "maps":
        inv = torch.fft.irfft2(torch.where(mult > 0, w0 / torch.where(mult > 0, mult, 1.0), 0.0), s=(n, n))
        return {"w": mult * torch.fft.rfft2(s), "s": inv}
    P = _Plain(c, dev)

    def probes(w, px):
        st = n // px
        u, v = _velocity(w, n)
        return torch.stack([u[:, ::st, ::st].flatten(1), v[:, ::st, ::st].flatten(1)], dim=-1)

    def window(w, steps, px):
        out = [probes(w, px)] if c["t0"] else []
        for k in range(1, steps + 1):
            w = P.step(w)
            if k % c["every"] == 0:
                out.append(probes(w, px))
        return w, torch.stack(out, dim=1)

    if c["kind"] == "forward":
        w, obs = window(mult * torch.fft.rfft2(s), c["nsteps"], c["px"])
        return {"w": w, "obs": obs}
    if c["kind"] == "spectra":
        K = (n - 1) // 3
        nshell = int(math.sqrt(2.0) * K) + 1
        kept = (P.keep > 0) & (P.k2 > 0)
        shell = P.k2.sqrt().floor().long()[kept]
        wgt = (torch.where(P.kx == 0, 1.0, 2.0) * P.k2 / (2.0 * n ** 4))[kept]

        def shells(lam):
            out = torch.zeros(lam.shape[:-2] + (nshell,), device=dev, dtype=torch.float64)
            return out.index_add_(-1, shell, wgt * lam[..., kept].abs() ** 2)

        fields = [P.inv(mult * torch.fft.rfft2(s))]
        for _ in range(c["nsteps"] - 1):
            fields.append(P.inv(P.step(torch.fft.rfft2(fields[-1]) * P.keep)))
        lam = P.inv(lamT)
        member, mean = [], []

        def save():
            h = torch.fft.rfft2(lam)
            member.append(shells(h))
            mean.append(shells(h.mean(dim=0)))

        save()
        for k in range(c["nsteps"] - 1, -1, -1):
            x = fields[k].requires_grad_(True)
            (lam,) = torch.autograd.grad(P.inv(P.step(torch.fft.rfft2(x) * P.keep)), x, lam)
            fields[k] = None
            if k % c["every"] == 0:
                save()
        lam0 = torch.fft.rfft2(lam) * P.keep
        return {"member": torch.stack(member, dim=1), "mean": torch.stack(mean, dim=0), "lam0": lam0,
                "filtered": P.inv(mult * lam0)}
    x = s.clone().requires_grad_(True)
    w = mult * torch.fft.rfft2(x)
    if c["kind"] == "ragged":
        J, all_nu, all_f = [], P.nu, P.f
        for b, (steps, px, _, _) in enumerate(wins):
            P.nu, P.f = all_nu[b:b + 1], all_f[b:b + 1]
            _, obs = window(w[b:b + 1], steps, px)
            J.append(0.5 * (obs[0] - data[b]).square().sum())
        J = torch.stack(J)
    else:
        w, obs = window(w, c["nsteps"], c["px"])
        J = 0.5 * (obs - torch.stack(data)).square().sum(dim=(1, 2, 3))
    (g,) = torch.autograd.grad(J.sum(), x)
    if c["kind"] == "autograd":
        return {"obs": obs.detach(), "w": w.detach(), "loss": J.sum().detach(), "grad": g}
    return {"J": J.detach(), "grad": g}
