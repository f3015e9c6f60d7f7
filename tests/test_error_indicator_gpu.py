"""The a-posteriori error indicator ||psi|| b_m |c_{m-1}| of the report where c_{m-1} is far below 1e-19, so that
its square is below FP32's range.  One fidelity-only slice; expected: the oracle's Lanczos coefficients and the
Taylor series of exp(-i dt T) e_1, whose last entry has no cancellation.  Tolerance 1 %: FP32 arithmetic on the
indicator, FP64 (or float-float) Lanczos coefficients, up to 16 of which enter as a product.  (Float-float on the
smaller couplings only: with Jz = 60 the recurrence amplifies the vectors' 44 bits to some per cent of the last
coefficients.)"""
import numpy as np
import pytest
import torch

import oracle
import oracle.sector as S
from oracle.krylov import lanczos
from paper_2010_03598_gb300 import workloads as W

pytestmark = pytest.mark.gpu
U = 0.3


def expected(apply_H, psi, m, dt):
    _, a, b, bm, _, broke = lanczos(apply_H, psi, m)
    assert not broke
    T = np.diag(a) + np.diag(b, 1) + np.diag(b, -1)
    y = np.zeros(m, complex)
    y[0] = 1.0
    c = y.copy()
    for k in range(1, 41):
        y = (-1j * dt / k) * (T @ y)
        c += y
    return bm * abs(c[-1])


@pytest.mark.parametrize("prec,Jxy,Jz,m,dt", [("c128", 0.2, 60.0, 16, 0.03), ("c128", 0.5, 20.0, 12, 0.01),
                                               ("ff", 0.5, 20.0, 12, 0.01)])
def test_subspace(prec, Jxy, Jz, m, dt):
    from paper_2010_03598_gb300 import api as A
    c = S.SectorChain(10, 4, 1, Jxy, Jz, 1 | 512, 1.0)
    psi = np.zeros(c.D, complex)
    psi[0] = 1.0
    eng = A.KGrapeSector(A.SectorSpec(10, 4, 1, Jxy, Jz), A.Options(1, dt, m, prec=prec, grad="none"))
    t = torch.tensor(psi).cuda()
    eng.evaluate(torch.tensor([[U]], dtype=torch.float64).cuda(), t, t)
    got = eng.sync()["krylov_err_max"]
    eng.close()
    want = expected(lambda v: c.apply_H(U, v), psi, m, dt)
    print(prec, got, want)
    assert want < 1e-23 and abs(got - want) <= 0.01 * want


@pytest.mark.parametrize("kw", [dict(), dict(tile_bits=6, ctas=4)])
def test_chain(kw):
    from paper_2010_03598_gb300 import api as A
    L, Jxy, Jz, m, dt = 8, 0.05, 20.0, 12, 0.01
    c = oracle.Chain(L, Jxy, Jz, "sz", hc_mask=1 | 128, hc_amp=1.0)
    psi = W.neel_state(L).astype(complex)
    eng = A.KGrape(A.ChainSpec(L, Jxy, Jz, hc_kind="sz", hc_mask=1 | 128), A.Options(1, dt, m, prec="c128", grad="none", **kw))
    t = torch.tensor(psi).cuda()
    eng.evaluate(torch.tensor([U], dtype=torch.float64).cuda(), t, t)
    got = eng.sync()["krylov_err_max"]
    eng.close()
    want = expected(lambda v: c.apply_H(U, v), psi, m, dt)
    print(got, want)
    assert want < 1e-23 and abs(got - want) <= 0.01 * want
