"""Performance cases of the K-GRAPE library: what a program that optimises pulses has it do.

A case is one evaluation (fidelity, and the gradient unless it says "none") through the public entry
points, over the range that programs use: pulses on chains of a few to 24 spins, a batch of pulses in
one launch, and the parity-excitation subspaces of the paper; complex64, complex128 and float-float
vectors; every gradient mode in use; checkpointed and fully stored trajectories.

The pulse is a torch tensor in the type in which a program keeps such parameters: float32 (torch's
default) with a complex64 engine, whose results carry single precision, and float64 with the
complex128 and float-float engines.  The library's interface is float64 throughout; what comes back
goes to the pulse's type, as autograd does it for a parameter.
"""
from __future__ import annotations

import itertools
import math

import numpy as np
import torch

from paper_2010_03598_gb300 import api
from paper_2010_03598_gb300 import workloads as W

C128 = torch.complex128


# ---------------------------------------------------------------- the cases
def listed():
    return [
        # One pulse on the smallest chain of the workloads: a call of a few milliseconds, latency only.
        chain("pulse 8 spins", L=8, N=64, m=12, dt=0.1, Jz=0.5),
        # The paper's control operator (Sz on both ends), zeroth-order gradient, sizes that are no powers of two.
        chain("pulse 11 spins, Sz control", L=11, N=77, m=13, dt=0.07, Jz=1.3, hc="sz", grad="zeroth"),
        # The exact (Gauss-Lobatto) gradient, for large time steps.
        chain("pulse 14 spins, exact gradient", L=14, N=60, m=16, dt=0.1, Jz=0.8, grad="exact"),
        # The 16-spin workload.
        chain("pulse 16 spins", L=16, N=200, m=20, dt=0.05, Jz=1.0),
        # A line search evaluates F alone: the forward direction.
        chain("fidelity only 18 spins", L=18, N=90, m=18, dt=0.05, Jz=0.5, grad="none"),
        # The benchmark's chain and basis, a quarter of its pulse.
        chain("pulse 20 spins", L=20, N=100, m=20, dt=0.05, Jz=0.5),
        # The longest chain of the workloads: checkpoints and recomputation.
        chain("pulse 24 spins, checkpoints", L=24, N=8, m=24, dt=0.05, Jz=0.5, ckpt=4),
        # The complex128 engine: reference results, tight convergence.
        chain("double 16 spins", L=16, N=25, m=20, dt=0.05, Jz=1.0, prec="c128"),
        # The batch workload's 256 pulses of 10 to 16 spins in one launch (random restarts, parameter scans).
        batch("batch of 256 pulses", B=256, Lmin=10, Lmax=16, N=40, m=16, dt=0.05),
        # The paper's own task, 14 spins and 4 excitations (D = 511): as many pulses as the card holds at once.
        sector("subspace 14 spins, 1216 pulses", L=14, K=4, B=1216, N=128, m=10, dt=0.5),
        # The same task on 20 spins (D = 2445) in float-float vectors, which its long pulses need.
        sector("subspace 20 spins, float-float", L=20, K=4, B=152, N=32, m=10, dt=0.5, prec="ff"),
        # One pulse of the paper's smallest task (D = 110, N = 4 D) in complex128: an L-BFGS step.
        sector("subspace 10 spins, one pulse", L=10, K=4, B=1, N=440, m=10, dt=0.5, prec="c128"),
    ]


def chain(name, *, L, N, m, dt, Jz, hc="sx", grad="centered", prec="c64", ckpt=0):
    return dict(name=name, kind="chain", L=L, N=N, m=m, dt=dt, Jz=Jz, hc=hc, grad=grad, prec=prec, ckpt=ckpt)


def batch(name, *, B, Lmin, Lmax, N, m, dt):
    return dict(name=name, kind="batch", B=B, Lmin=Lmin, Lmax=Lmax, N=N, m=m, dt=dt, prec="c64")


def sector(name, *, L, K, B, N, m, dt, parity=1, grad="centered", prec="c64"):
    return dict(name=name, kind="sector", L=L, K=K, parity=parity, B=B, N=N, m=m, dt=dt, grad=grad, prec=prec)


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["chain"] * 5 + ["chain128"] * 2 + ["batch"] + ["sector"] * 3)
    if kind == "chain":
        L, m = rng.randint(5, 22), rng.randint(8, 24)
        step_us = 6.0 if L <= 18 else 9.0 * 4.0 ** max(0, L - 20)  # an upper estimate of a Lanczos step
        N = _log_int(rng, 8, max(9, min(256, 0.1e6 / (2 * m * step_us))))
        grad = rng.choice(["centered", "centered", "zeroth", "exact", "none"])
        c = chain("", L=L, N=N, m=m, dt=round(rng.uniform(0.03, 0.1), 3), Jz=round(rng.uniform(0.0, 2.0), 2),
                  hc=rng.choice(["sx", "sx", "sz"]), grad=grad,
                  ckpt=rng.choice([0, 0, max(2, math.isqrt(N))]) if grad != "exact" else 0)
    elif kind == "chain128":
        L, m = rng.randint(5, 18), rng.randint(8, 24)
        N = _log_int(rng, 6, 100 if L <= 14 else 24)
        c = chain("", L=L, N=N, m=m, dt=round(rng.uniform(0.03, 0.1), 3), Jz=round(rng.uniform(0.0, 2.0), 2),
                  hc=rng.choice(["sx", "sz"]), grad=rng.choice(["centered", "none"]), prec="c128")
    elif kind == "batch":
        Lmin = rng.randint(8, 13)
        c = batch("", B=_log_int(rng, 16, 256), Lmin=Lmin, Lmax=min(16, Lmin + rng.randint(0, 6)),
                  N=rng.randint(8, 32), m=rng.randint(10, 20), dt=round(rng.uniform(0.03, 0.08), 3))
    else:
        L, K = rng.choice([(8, 3), (10, 4), (11, 5), (12, 4), (12, 6), (13, 5), (14, 4), (15, 4), (17, 4), (20, 4)])
        c = sector("", L=L, K=K, parity=rng.choice([1, 1, -1]), B=_log_int(rng, 1, 608), N=rng.randint(16, 64),
                   m=rng.randint(10, 14), dt=round(rng.uniform(0.2, 0.5), 2), grad=rng.choice(["centered", "zeroth"]),
                   prec=rng.choice(["c64", "ff", "c128"]))
    del c["name"]
    return c


# ---------------------------------------------------------------- a program's state before the call
def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _normal(gen, *shape):
    return torch.complex(torch.randn(*shape, generator=gen, device="cuda", dtype=torch.float64),
                         torch.randn(*shape, generator=gen, device="cuda", dtype=torch.float64))


def _unit(f):
    return f / torch.linalg.vector_norm(f, dim=-1, keepdim=True)


def _controls(case, gen, *shape):
    dtype = torch.float32 if case["prec"] == "c64" else torch.float64
    return torch.rand(*shape, generator=gen, device="cuda", dtype=dtype) * 2 - 1  # u ~ U(-1, 1)


def _mask(L):  # an Sz control's sites: both ends, as in the paper's (J/2)(sigma^z_1 + sigma^z_L)
    return 1 | 1 << (L - 1)


def _neel(L):
    psi = torch.zeros(1 << L, dtype=C128, device="cuda")
    psi[W.neel_index(L)] = 1
    return psi


def _target(gen, L, hc, Jz, u, dt):
    """Targets [n, 2^L] that the pulses u [n, N] partly reach, as in an optimisation that is under way: the Neel state
    carried over a shifted pulse by a coarse product formula (steps of about 0.25), plus a random part."""
    n, N = u.shape
    u = u + min(0.5, 1.5 / (N * dt))
    k = max(1, int(0.25 / dt))
    psi = _neel(L).repeat(n, 1)
    for j0 in range(0, N, k):
        tau = dt * min(k, N - j0)
        theta = 0.5 * dt * u[:, j0:j0 + k].double().sum(1)
        if hc == "sx":  # exp(-i theta sigma_x) on site 1
            v = psi.view(n, -1, 2)
            c, s = torch.cos(theta).view(n, 1, 1), -1j * torch.sin(theta).view(n, 1, 1)
            psi = (c * v + s * v.flip(2)).reshape(n, -1)
        else:  # exp(-i theta sigma_z) on the sites of the mask
            for site in (0, L - 1):
                v = psi.view(n, -1, 2, 1 << site)
                v *= torch.stack([torch.exp(-1j * theta), torch.exp(1j * theta)], 1).view(n, 1, 2, 1)
        zz = torch.exp(-1j * tau * Jz / 4).view(n, 1, 1)
        for b in range(L - 1):  # bond b: exp(-i tau h_b) on bits b, b + 1
            v = psi.view(n, -1, 2, 2, 1 << b)
            x, y = v[:, :, 0, 1].clone(), v[:, :, 1, 0].clone()
            v *= zz.view(n, 1, 1, 1, 1)
            c, s = math.cos(tau / 2), -1j * math.sin(tau / 2)
            v[:, :, 0, 1] = (c * x + s * y) * zz.conj()
            v[:, :, 1, 0] = (c * y + s * x) * zz.conj()
    return _unit(psi + 0.3 * _unit(_normal(gen, n, 1 << L)))


def _spec(case, L, Jz):
    return api.ChainSpec(L, 1.0, float(Jz), hc_kind=case.get("hc", "sx"), hc_mask=_mask(L) if case.get("hc") == "sz" else 0)


def _batch_draw(case, seed):
    r = np.random.default_rng(seed)
    Ls = np.sort(r.integers(case["Lmin"], case["Lmax"] + 1, case["B"]))  # grouped by length: made group by group
    return Ls, r.uniform(0.0, 2.0, case["B"])


def _inputs(case, seed):
    """The plain inputs of a case: what prepare() binds an engine to, and what exact() works from."""
    gen = _generator(seed)
    if case["kind"] == "chain":
        u = _controls(case, gen, case["N"])
        Jz = torch.full((1,), case["Jz"], dtype=torch.float64, device="cuda")
        return dict(u=u, psi0=_neel(case["L"]), target=_target(gen, case["L"], case["hc"], Jz, u[None], case["dt"])[0])
    if case["kind"] == "batch":
        Ls, deltas = _batch_draw(case, seed)
        u = _controls(case, gen, case["B"], case["N"])
        psi0, target = [], []
        for L in np.unique(Ls):
            at = np.flatnonzero(Ls == L)
            f = _target(gen, int(L), "sx", torch.tensor(deltas[at], device="cuda"), u[at[0]:at[-1] + 1], case["dt"])
            target += list(f.unbind(0))
            psi0 += [_neel(int(L))] * len(at)
        return dict(u=u, psi0=psi0, target=target, Ls=Ls, deltas=deltas)
    D = len(_sector_states(case))
    u = _controls(case, gen, case["B"], case["N"])
    psi0 = torch.zeros(D, dtype=C128, device="cuda")  # the paper's task e_1 -> e_D
    target = psi0.clone()
    psi0[0] = 1
    target[D - 1] = 1
    return dict(u=u, psi0=psi0, target=target)


def prepare(case, seed):
    s = dict(_inputs(case, seed), case=case)
    if case["kind"] == "chain":
        opts = api.Options(case["N"], case["dt"], case["m"], prec=case["prec"], grad=case["grad"], ckpt_every=case["ckpt"])
        s["engine"] = api.KGrape(_spec(case, case["L"], case["Jz"]), opts)
        s["u"].requires_grad_(case["grad"] != "none")
    elif case["kind"] == "batch":
        opts = api.Options(case["N"], case["dt"], case["m"], prec="c64")
        s["u64"] = s["u"].double()  # the launch reads the pulses here
        s["engine"] = api.KGrapeBatch([_spec(case, int(L), d) for L, d in zip(s["Ls"], s["deltas"])], opts,
                                      list(s["u64"].unbind(0)), s["psi0"], s["target"])
    else:
        spec = api.SectorSpec(case["L"], case["K"], case["parity"])
        opts = api.Options(case["N"], case["dt"], case["m"], prec=case["prec"], grad=case["grad"])
        s["engine"] = api.KGrapeSector(spec, opts, B=case["B"])
    return s


# ---------------------------------------------------------------- one pass
def run(s):
    u, kind = s["u"], s["case"]["kind"]
    if kind == "chain" and s["case"]["grad"] == "none":  # a line search's trial point
        fid, _ = s["engine"].evaluate(u.double(), s["psi0"], s["target"])
        return {"F": fid.to(u.dtype)}
    if kind == "chain":  # a step of gradient ascent on F, up to the optimiser
        F = api.fidelity(u.double(), s["engine"], s["psi0"], s["target"]).to(u.dtype)
        grad, = torch.autograd.grad(F, u, torch.ones_like(F))
        return {"F": F.detach(), "grad": grad}
    if kind == "batch":
        s["u64"].copy_(u)
        s["engine"].launch()
        fid, grad = s["engine"].fid, s["engine"].grads
    else:
        fid, grad = s["engine"].evaluate(u.double(), s["psi0"], s["target"])
    return {"F": fid.to(u.dtype), "grad": grad.to(u.dtype)}


# ---------------------------------------------------------------- what a pass cannot do without
def work(case):
    """Inputs read and outputs written once; the real operations of the Krylov evaluation itself (per amplitude and
    Lanczos step: one complex addition per antiparallel bond, half of the bonds on average, the diagonal, the
    two-term recurrence and its sums, about 28 more; per slice 8 m for the recombination)."""
    if case["kind"] == "batch":
        Ls, _ = _batch_draw(case, 0)
        parts = [work(chain("", L=int(L), N=case["N"], m=case["m"], dt=case["dt"], Jz=1.0)) for L in Ls]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    N, m, B = case["N"], case["m"], case.get("B", 1)
    if case["kind"] == "chain":
        D, bonds = 1 << case["L"], case["L"] - 1
    else:
        D, bonds = len(_sector_states(case)), 2 * case["K"] * (case["L"] - case["K"]) / case["L"]
    slices = N if case["grad"] == "none" else 2 * N
    recombinations = 3 if case["grad"] == "exact" else 1
    flops = float(slices) * D * (m * ((bonds if case["kind"] == "chain" else 2 * bonds) + 28) + 8 * m * recombinations) * B
    return {"bytes": 32.0 * D + B * (8.0 * N + 8.0 + (8.0 * N if case["grad"] != "none" else 0.0)), "flops": flops}


# ---------------------------------------------------------------- the same in 64 bits, plain torch
class _Chain:
    """H = H0 + u Hc on vectors [n, 2^L], the pulses' Jz [n]."""

    def __init__(self, L, hc, Jz):
        self.L, self.hc = L, hc
        i = torch.arange(1 << L, device="cuda")
        par = sum((1 - 2 * ((i >> b ^ i >> b + 1) & 1) for b in range(L - 1)), torch.zeros_like(i))
        self.diag = Jz.view(-1, 1) * (0.25 * par)
        self.z = 0.5 * sum(1 - 2 * (i >> s & 1) for s in range(L) if _mask(L) >> s & 1)
        self.bound = (L - 1) * (0.5 + 0.25 * float(Jz.abs().max())) + 1.0

    def hc_apply(self, v):
        return 0.5 * v.view(v.shape[0], -1, 2).flip(2).reshape(v.shape) if self.hc == "sx" else self.z * v

    def apply(self, v, u):
        out = self.diag * v
        for b in range(self.L - 1):
            x, y = v.view(v.shape[0], -1, 2, 2, 1 << b), out.view(v.shape[0], -1, 2, 2, 1 << b)
            y[:, :, 0, 1].add_(x[:, :, 1, 0], alpha=0.5)
            y[:, :, 1, 0].add_(x[:, :, 0, 1], alpha=0.5)
        return out.addcmul_(u.to(C128).view(-1, 1), self.hc_apply(v))


def _mirror(s, L):
    return int(format(s, "0%db" % L)[::-1], 2)


def _sector_states(case):
    """The smaller member of every mirror orbit of the K-excitation states, ascending (without palindromes for parity -1)."""
    L, K = case["L"], case["K"]
    states = [sum(1 << k for k in sites) for sites in itertools.combinations(range(L), K)]
    return sorted(s for s in states if s < _mirror(s, L) or s == _mirror(s, L) and case["parity"] == 1)


class _Sector:
    """The same in the parity-excitation subspace (J = 1, alpha_z = 0.5 of the paper: Jxy = 2, Jz = 1)."""

    def __init__(self, case):
        L, p, states = case["L"], case["parity"], _sector_states(case)
        row = {s: r for r, s in enumerate(states)}
        cols, wgts = [], []
        for s in states:
            n, c, w = 1 if _mirror(s, L) == s else 2, [], []
            for b in range(L - 1):
                if (s >> b ^ s >> b + 1) & 1:
                    t = s ^ 3 << b
                    q = min(t, _mirror(t, L))
                    if q in row:
                        c.append(row[q])
                        w.append((1.0 if q == t else p) * math.sqrt(n / (1 if _mirror(q, L) == q else 2)))
            cols.append(c)
            wgts.append(w)
        width = max(map(len, cols))
        self.cols = torch.tensor([c + [0] * (width - len(c)) for c in cols], device="cuda").T.contiguous()
        self.wgts = torch.tensor([w + [0.0] * (width - len(w)) for w in wgts], device="cuda", dtype=torch.float64).T.contiguous()
        s = torch.tensor(states, device="cuda")
        self.diag = 0.25 * sum(1 - 2 * ((s >> b ^ s >> b + 1) & 1) for b in range(L - 1))
        self.z = 0.5 * sum(1 - 2 * (s >> k & 1) for k in (0, L - 1))
        self.bound = 0.25 * (L - 1) + float(self.wgts.abs().sum(0).max()) + 1.0

    def hc_apply(self, v):
        return self.z * v

    def apply(self, v, u):
        out = (self.diag + u.view(-1, 1) * self.z) * v
        for c, w in zip(self.cols, self.wgts):
            out.addcmul_(v[:, c], w)
        return out


def _exp(H, v, u, tau):
    """exp(-i tau H) v by the Taylor series, in steps with |tau| ||H|| <= 2."""
    steps = max(1, math.ceil(abs(tau) * H.bound / 2))
    r = abs(tau) * H.bound / steps
    for _ in range(steps):
        term, out, size, k = v, v.clone(), 1.0, 0
        while size > 1e-18:
            k += 1
            size *= r / k
            term = H.apply(term, u) * (-1j * tau / steps / k)
            out += term
        v = out
    return v


def _overlap(x, y):
    return (x.conj() * y).sum(-1)


def _evaluate(H, u, psi0, target, dt, grad):
    """F [n] and dF/du [n, N] of the pulses u [n, N] with exact slice propagators: G(t) = 2 dt Im <chi(t)|Hc|psi(t)>
    at the slice ends (zeroth order: at its end; centred: the mean of both) and, for the exact gradient, at the nodes
    of the 4-point Gauss-Lobatto rule."""
    N = u.shape[1]
    nodes = [0.5 * dt * (1 - 1 / math.sqrt(5)), 0.5 * dt * (1 + 1 / math.sqrt(5))]
    psi, inner = [psi0.expand(u.shape[0], -1)], []
    for j in range(N):
        if grad == "exact":
            inner.append([_exp(H, psi[-1], u[:, j], s) for s in nodes])
        psi.append(_exp(H, psi[-1], u[:, j], dt))
    beta = _overlap(target, psi[-1])
    F = beta.abs() ** 2
    if grad == "none":
        return F, None
    chi = beta[:, None] * target
    g = lambda x, y: 2 * dt * _overlap(x, H.hc_apply(y)).imag  # noqa: E731
    G = [None] * N + [g(chi, psi[N])]
    out = torch.empty(u.shape, dtype=torch.float64, device="cuda")
    for j in range(N - 1, -1, -1):
        mid = 0.0
        if grad == "exact":
            mid = sum(g(_exp(H, chi, u[:, j], s - dt), inner[j][k]) for k, s in enumerate(nodes))
        chi = _exp(H, chi, u[:, j], -dt)
        G[j] = g(chi, psi[j])
        out[:, j] = G[j + 1] if grad == "zeroth" else 0.5 * (G[j] + G[j + 1]) if grad == "centered" else (G[j] + G[j + 1]) / 12 + 5 * mid / 12
    return F, out


def exact(case, seed):
    s = _inputs(case, seed)
    if case["kind"] == "chain":
        H = _Chain(case["L"], case["hc"], torch.full((1,), case["Jz"], dtype=torch.float64, device="cuda"))
        F, grad = _evaluate(H, s["u"].double()[None], s["psi0"], s["target"][None], case["dt"], case["grad"])
        return {"F": F} if grad is None else {"F": F, "grad": grad[0]}
    if case["kind"] == "batch":
        F, grad = [], []
        for L in np.unique(s["Ls"]):
            at = np.flatnonzero(s["Ls"] == L)
            H = _Chain(int(L), "sx", torch.tensor(s["deltas"][at], device="cuda"))
            f, g = _evaluate(H, s["u"][at[0]:at[-1] + 1].double(), _neel(int(L)), torch.stack(s["target"][at[0]:at[-1] + 1]),
                             case["dt"], "centered")
            F.append(f)
            grad.append(g)
        return {"F": torch.cat(F), "grad": torch.cat(grad)}
    F, grad = _evaluate(_Sector(case), s["u"].double(), s["psi0"], s["target"][None], case["dt"], case["grad"])
    return {"F": F, "grad": grad}
