"""The kernel that holds one tile of amplitudes per CTA in registers, against the oracle.

It serves single evaluations whose schedule is left to the library on short chains.  Sizes: every
block shape (chains with fewer amplitudes than a warp, one warp, several, the largest), every bond
position and control site that has code of its own, basis sizes around the switch between shared
and global memory, breakdowns, an invariant subspace, checkpoints and every gradient mode.
Tolerances are those of test_parity_gpu.py: 1e-10 (complex128), 1e-5 / 1e-4 (complex64).
"""
import numpy as np
import pytest
import torch

import oracle
from paper_2010_03598_gb300 import workloads as W

pytestmark = pytest.mark.gpu
TOL = {"c128": (1e-10, 1e-10), "c64": (1e-5, 1e-4)}


def evaluate(spec, opts, u, psi0, f):
    from paper_2010_03598_gb300 import api as A
    dev = torch.device("cuda", 0)
    eng = A.KGrape(A.ChainSpec(**spec), A.Options(**opts))
    fid, grad = eng.evaluate(torch.tensor(u, device=dev), torch.tensor(psi0, device=dev), torch.tensor(f, device=dev))
    rep = eng.sync()
    out = float(fid.item()), (grad.cpu().numpy().copy() if opts["grad"] != "none" else None), rep
    eng.close()
    return out


def problem(L, N, seed, hc):
    rng = np.random.default_rng(seed)
    u = rng.uniform(-1, 1, N)
    # a target with a healthy overlap: relative errors are then those of the arithmetic (complex64
    # rounding of an overlap far below a typical one would be amplified)
    psi0 = rng.standard_normal(1 << L) + 1j * rng.standard_normal(1 << L)
    psi0 /= np.linalg.norm(psi0)
    f = psi0 + 0.8 * W.draw_target(rng, 1 << L)
    f /= np.linalg.norm(f)
    spec = dict(L=L, Jxy=1.0, Jz=0.7, hc_amp=0.9)
    if hc == "sz":
        mask = 1 | (1 << (L - 1))
        return u, psi0, f, dict(spec, hc_kind="sz", hc_mask=mask), oracle.Chain(L, 1.0, 0.7, "sz", hc_mask=mask, hc_amp=0.9)
    return u, psi0, f, dict(spec, hc_site=hc), oracle.Chain(L, 1.0, 0.7, "sx", hc_site=hc, hc_amp=0.9)


def check(prec, F, g, F_ref, g_ref):
    assert abs(F - F_ref) <= TOL[prec][0] * abs(F_ref), (F, F_ref)
    if g is not None:
        assert np.linalg.norm(g - g_ref) <= TOL[prec][1] * np.linalg.norm(g_ref)


CASES = [(L, hc, m, mode) for L, hc, m, mode in [
    (1, 0, 4, "centered"), (2, 1, 6, "exact"), (3, "sz", 8, "zeroth"), (4, 3, 12, "centered"), (5, 0, 1, "centered"),
    (5, 4, 20, "exact"), (6, 5, 9, "none"), (6, "sz", 16, "centered"), (7, 6, 13, "exact"), (7, 0, 32, "zeroth"),
    (8, 0, 12, "centered"), (8, 7, 32, "exact"), (8, 4, 2, "zeroth"), (9, 8, 20, "exact"), (9, "sz", 24, "centered"),
    (10, 0, 11, "exact"), (10, 9, 10, "zeroth"), (10, 6, 25, "none"), (11, "sz", 13, "exact"), (11, 10, 12, "centered"),
    (12, 0, 16, "exact"), (12, 11, 12, "centered"), (12, 8, 5, "zeroth")]]


@pytest.mark.parametrize("prec", ["c64", "c128"])
@pytest.mark.parametrize("L,hc,m,mode", CASES)
def test_every_block_shape_and_mode_vs_oracle(L, hc, m, mode, prec):
    N, dt = 7, 0.06
    u, psi0, f, spec, ch = problem(L, N, 700 + L, hc)
    F_ref, g_ref, _ = oracle.evaluate(ch, u, dt, m, psi0, f, "centered" if mode == "none" else mode)
    F, g, rep = evaluate(spec, dict(N=N, dt=dt, m=m, prec=prec, grad=mode), u, psi0, f)
    check(prec, F, g, F_ref, g_ref)
    assert rep["status"] == 0 and abs(rep["norm_final"] - 1.0) < (1e-12 if prec == "c128" else 1e-5)


@pytest.mark.parametrize("prec", ["c64", "c128"])
@pytest.mark.parametrize("L,hc,m,mode", [(13, 12, 9, "exact"), (14, 13, 6, "centered"), (14, 8, 7, "zeroth"), (15, "sz", 8, "zeroth"), (15, 7, 7, "none"),
                                         (14, 9, 8, "exact"), (15, 10, 8, "centered"),
                                         (16, 8, 8, "centered"), (16, 9, 6, "exact"), (17, 16, 6, "centered"), (18, 0, 6, "zeroth")])
def test_several_ctas_vs_oracle(L, hc, m, mode, prec):
    # 16 to 128 CTAs with one tile each: tiles of 128 to 2048 amplitudes, the control inside the tile, on
    # its top bit (complex128, L = 16: bit 8; complex64, L = 14: bit 8, L = 15: bit 9) and above it
    N, dt = 2, 0.05
    u, psi0, f, spec, ch = problem(L, N, 750 + L, hc)
    F_ref, g_ref, _ = oracle.evaluate(ch, u, dt, m, psi0, f, "centered" if mode == "none" else mode)
    F, g, rep = evaluate(spec, dict(N=N, dt=dt, m=m, prec=prec, grad=mode), u, psi0, f)
    check(prec, F, g, F_ref, g_ref)
    assert rep["status"] == 0 and rep["ctas"] > 1


@pytest.mark.parametrize("prec,L", [("c128", 12), ("c64", 14)])
def test_group_that_a_member_never_joins_times_out_cleanly(prec, L):
    # CTA 0 does not post its first sums (host-side fault injection): every wait runs out, the launch ends
    # with KG_ERR_TIMEOUT, and the next launch on the same engine is clean and deterministic.
    from paper_2010_03598_gb300 import _abi
    from paper_2010_03598_gb300 import api as A
    N = 3
    u, psi0, f, spec, ch = problem(L, N, 77, 0)
    dev = torch.device("cuda", 0)
    eng = A.KGrape(A.ChainSpec(**spec), A.Options(N, 0.05, 8, prec=prec))
    t = [torch.tensor(x, device=dev) for x in (u, psi0, f)]
    for kind in (1, 2):
        try:
            A.set_wait_limit_ns(50_000_000)
            _abi.check(_abi.lib().kg_debug_set_fault(kind), "kg_debug_set_fault")
            eng.evaluate(*t)
            with pytest.raises(_abi.KGrapeError) as ei:
                eng.sync()
            assert ei.value.status == _abi.KG_ERR_TIMEOUT
        finally:
            A.set_wait_limit_ns(2_000_000_000)
            _abi.lib().kg_debug_set_fault(0)
    got = []
    for _ in range(2):
        fid, grad = eng.evaluate(*t)
        assert eng.sync()["ctas"] > 1
        got.append((float(fid.item()), grad.cpu().numpy().copy()))
    eng.close()
    assert got[0][0] == got[1][0] and np.array_equal(got[0][1], got[1][1])
    F_ref, g_ref, _ = oracle.evaluate(ch, u, 0.05, 8, psi0, f, "centered")
    check(prec, *got[0], F_ref, g_ref)


@pytest.mark.parametrize("L,hc", [(13, 0), (14, 13), (15, "sz"), (16, 15), (17, 0), (18, 17)])
def test_exchange_by_messages_repeats_bit_for_bit(L, hc):
    """Every amplitude and every sum is used as it was sent, whenever it arrives: each evaluation gives the same bits."""
    u, psi0, f, spec, _ = problem(L, 12, 300 + L, hc)
    opts = dict(N=12, dt=0.1, m=16, prec="c64", grad="centered")
    F0, g0, _ = evaluate(spec, opts, u, psi0, f)
    for _ in range(5):
        F, g, _ = evaluate(spec, opts, u, psi0, f)
        assert F == F0 and np.array_equal(g, g0)


@pytest.mark.parametrize("prec", ["c64", "c128"])
@pytest.mark.parametrize("L,N,C", [(4, 9, 2), (8, 11, 4), (9, 6, 1), (11, 10, 9), (7, 5, 7), (14, 7, 3)])
def test_checkpoints_are_bitwise_equal_to_the_full_trajectory(L, N, C, prec):
    u, psi0, f, spec, ch = problem(L, N, 800 + L, 0)
    full = evaluate(spec, dict(N=N, dt=0.05, m=10, prec=prec, grad="centered"), u, psi0, f)
    part = evaluate(spec, dict(N=N, dt=0.05, m=10, prec=prec, grad="centered", ckpt_every=C), u, psi0, f)
    assert full[0] == part[0] and np.array_equal(full[1], part[1])
    F_ref, g_ref, _ = oracle.evaluate(ch, u, 0.05, 10, psi0, f, "centered")
    check(prec, full[0], full[1], F_ref, g_ref)


@pytest.mark.parametrize("prec", ["c64", "c128"])
@pytest.mark.parametrize("L", [6, 8, 11, 13])
def test_invariant_and_nearly_invariant_subspaces(L, prec):
    # |0...0> is an eigenstate of H0 and of the Sz control: the basis ends after one vector.  With 1 %
    # of a random state the identity for b_1 cancels, and b_1 is formed explicitly, in every slice.
    N, m, dt, D = 5, 10, 0.05, 1 << L
    u, psi0, f, spec, ch = problem(L, N, 900 + L, "sz")
    for share in (0.0, 0.01):
        p = share * psi0
        p[0] += 1.0
        p /= np.linalg.norm(p)
        g = 0.5 * psi0 + 0.1 * f
        g[0] += 1.0
        g /= np.linalg.norm(g)
        F_ref, g_ref, _ = oracle.evaluate(ch, u, dt, m, p, g, "centered")
        F, gr, rep = evaluate(spec, dict(N=N, dt=dt, m=m, prec=prec, grad="centered"), u, p, g)
        assert abs(F - F_ref) <= TOL[prec][0] * F_ref
        # G_j = 2 dt Im <chi|Hc|psi> is the imaginary part of an overlap of modulus below 1 (exactly 0 in
        # the eigenstate): its rounding is that of the overlap, held to the tolerance on F
        assert np.linalg.norm(gr - g_ref) <= TOL[prec][0] * 2 * dt * np.sqrt(N)
        assert rep["status"] == 0 and rep["breakdowns"] >= (N if share == 0.0 else 0)


@pytest.mark.parametrize("dt", [0.2, 0.5])
def test_subspace_norm_does_not_drift_in_complex64(dt):
    # 2000 slices on D = 28: FP32 rounding of the states walks by about 6e-8 per slice (sqrt(N) of it, x4 margin)
    import oracle.sector as OS
    from paper_2010_03598_gb300 import api as A
    c = OS.paper_chain(8, 3, 1)
    N = 2000
    rng = np.random.default_rng(5)
    psi0 = rng.standard_normal(c.D) + 1j * rng.standard_normal(c.D)
    psi0 /= np.linalg.norm(psi0)
    dev = torch.device("cuda", 0)
    eng = A.KGrapeSector(A.SectorSpec(8, 3, 1), A.Options(N, dt, 12, prec="c64", grad="none"), B=1)
    u = torch.tensor(rng.uniform(-1, 1, (1, N)), device=dev)
    p = torch.tensor(psi0, device=dev)
    eng.evaluate(u, p, p)
    rep = eng.sync()
    assert rep["status"] == 0
    assert abs(rep["norm_final"] - 1.0) <= 4 * 6e-8 * np.sqrt(N) + 1e-7
    eng.close()


@pytest.mark.parametrize("prec", ["c64", "c128"])
@pytest.mark.parametrize("L", [6, 9, 12, 14, 18])
@pytest.mark.parametrize("norm", [2.2, 4.2])
def test_checkpoints_are_bitwise_equal_for_any_norm(prec, L, norm):
    # The recomputed first slice starts from 1 / ||psi_0|| as the forward sweep took it: at these norms the
    # reciprocal of the stored norm rounds differently.
    rng = np.random.default_rng(int(norm))
    psi0 = rng.standard_normal(1 << L) + 1j * rng.standard_normal(1 << L)
    psi0 *= norm / np.linalg.norm(psi0)
    u, _, f, spec, _ = problem(L, 8, 3, 0)
    full = evaluate(spec, dict(N=8, dt=0.05, m=10, prec=prec, grad="centered"), u, psi0, f)
    ckpt = evaluate(spec, dict(N=8, dt=0.05, m=10, prec=prec, grad="centered", ckpt_every=3), u, psi0, f)
    assert full[0] == ckpt[0] and np.array_equal(full[1], ckpt[1])
