"""The resident complex64 loop (4096-amplitude tiles on chip) against the oracle.

Chains of up to 18 spins reach it with an explicit schedule, 19 spins by default.  Covered: one and two tiles
per CTA; an Sx control in every place its partner is fetched from (inside an amplitude pair, in the tile, at
the tile's top bit, in another tile) and an Sz control; the gradient modes; bases shorter than the
recombination's copy ring; checkpoints.  Tolerances as in test_parity_gpu.py: 1e-5 on F, 1e-4 on the gradient.
"""
import numpy as np
import pytest
import torch

import oracle
from paper_2010_03598_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def problem(L, N, hc):
    rng = np.random.default_rng([L, 0 if hc == "sz" else 1 + hc])
    u = rng.uniform(-1, 1, N)
    psi0 = W.draw_target(rng, 1 << L)
    f = psi0 + 0.8 * W.draw_target(rng, 1 << L)  # a healthy overlap
    f /= np.linalg.norm(f)
    spec = dict(L=L, Jxy=1.0, Jz=0.7, hc_amp=0.9)
    if hc == "sz":
        mask = 1 | (1 << (L - 1))
        return u, psi0, f, dict(spec, hc_kind="sz", hc_mask=mask), oracle.Chain(L, 1.0, 0.7, "sz", hc_mask=mask, hc_amp=0.9)
    return u, psi0, f, dict(spec, hc_site=hc), oracle.Chain(L, 1.0, 0.7, "sx", hc_site=hc, hc_amp=0.9)


def evaluate(spec, u, psi0, f, dt, m, **opts):
    from paper_2010_03598_gb300 import api as A
    dev = torch.device("cuda", 0)
    eng = A.KGrape(A.ChainSpec(**spec), A.Options(len(u), dt, m, prec="c64", **opts))
    fid, grad = eng.evaluate(torch.tensor(u, device=dev), torch.tensor(psi0, device=dev), torch.tensor(f, device=dev))
    rep = eng.sync()
    out = float(fid.item()), grad.cpu().numpy().copy(), rep
    eng.close()
    return out


def check(L, ctas, hc, grad="centered", m=10, N=4, dt=0.05, default=False, **opts):
    u, psi0, f, spec, chain = problem(L, N, hc)
    schedule = {} if default else dict(tile_bits=12, ctas=ctas)
    F, g, rep = evaluate(spec, u, psi0, f, dt, m, grad=grad, **schedule, **opts)
    assert rep["threads"] == 544 and rep["ctas"] == ctas and rep["tile_bits"] == 12
    F_ref, g_ref, _ = oracle.evaluate(chain, u, dt, m, psi0, f, grad)
    ef, eg = abs(F - F_ref) / F_ref, np.linalg.norm(g - g_ref) / np.linalg.norm(g_ref)
    print(L, ctas, hc, grad, m, "rel. err F", ef, "grad", eg)
    assert ef <= 1e-5 and eg <= 1e-4, (ef, eg)
    return F, g


@pytest.mark.parametrize("L,ctas,hc", [(13, 1, 1), (13, 2, 12), (14, 2, 5), (14, 2, 11), (14, 4, 12), (14, 4, 13),
                                       (15, 4, 0), (15, 4, 1), (15, 4, 14), (15, 8, 11), (15, 8, "sz")])
def test_control_in_every_place(L, ctas, hc):
    check(L, ctas, hc)


@pytest.mark.parametrize("L,ctas,hc,grad", [(14, 2, 5, "exact"), (14, 4, 13, "exact"), (15, 4, "sz", "exact"),
                                            (14, 2, 12, "zeroth")])
def test_gradient_modes(L, ctas, hc, grad):
    check(L, ctas, hc, grad, m=12)


@pytest.mark.parametrize("ctas", [2, 4])
@pytest.mark.parametrize("m", [1, 2, 3, 4])
def test_bases_shorter_than_the_copy_ring(ctas, m):
    check(14, ctas, 12, m=m)


@pytest.mark.parametrize("ctas", [2, 4])
def test_checkpoints(ctas):
    L, N, hc = 14, 7, 13
    F, g = check(L, ctas, hc, N=N, ckpt_every=3)
    u, psi0, f, spec, _ = problem(L, N, hc)
    F0, g0, _ = evaluate(spec, u, psi0, f, 0.05, 10, tile_bits=12, ctas=ctas)
    assert F == F0 and np.array_equal(g, g0)


@pytest.mark.parametrize("hc,grad", [(0, "centered"), (13, "centered"), (5, "exact")])
def test_nineteen_spins_by_default(hc, grad):
    check(19, 128, hc, grad, m=8, N=2, default=True)
