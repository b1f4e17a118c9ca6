"""The float-float dielectric solve on the tensor cores (GW_F32X2, csrc/digit_screen.cu) against the oracle's
linear solve: one block of 32, whole and half last blocks of 64 rows, rows that end inside a 128-row tile.
Tolerance: NI float-float rounding errors of 2^-44 amplified by the condition number (< 100 here)."""
import numpy as np
import pytest

import gwinputs as gi
import oracle as orc

pytestmark = pytest.mark.gpu


def _ctx(ni, nq, nnu, v=None):
    import torch

    import paper_1602_02313_gb300 as gw
    from paper_1602_02313_gb300 import build as b
    b.build()
    cr = gi.make_crystal(ni, 1, 1, 1, ni, 60.0, qlist=[0] * nq)
    if v is not None:
        cr.v[:] = v
    gr = gi.make_grid(60.0, nnu, nnu, nnu, ncont=8)
    return torch, gw, cr, gw.GW(gr, cr, M=torch.zeros(nq, 1, ni, 1, 1, dtype=torch.complex128, device="cuda"))


@pytest.mark.parametrize("ni,nq,nnu", [(32, 2, 8), (64, 1, 8), (96, 3, 8), (160, 1, 8), (256, 2, 8), (288, 1, 8)])
def test_screen_digits(ni, nq, nnu):
    torch, gw, cr, ctx = _ctx(ni, nq, nnu)
    rng = np.random.default_rng(ni)
    X = (rng.standard_normal((nq, nnu, ni, ni)) + 1j * rng.standard_normal((nq, nnu, ni, ni))) / np.sqrt(2 * ni)
    Y = (rng.standard_normal((nq, nnu, ni, ni)) + 1j * rng.standard_normal((nq, nnu, ni, ni))) / np.sqrt(2 * ni)
    P = -0.02 * (X @ np.conj(np.swapaxes(X, -1, -2))) + 0.004 * (Y - np.conj(np.swapaxes(Y, -1, -2)))
    W = torch.full((nq, nnu, ni, ni), float("nan"), dtype=torch.complex128, device="cuda")
    info = torch.full((nq, nnu), -7, dtype=torch.int32, device="cuda")
    ctx.screen(0, nq, torch.from_numpy(P).cuda(), W, info, gw.GW_F32X2)
    ctx.sync()
    assert int(info.abs().sum()) == 0
    for q in range(nq):
        ref = orc.screen(P[q], cr.v[q])
        sv = np.sqrt(cr.v[q])
        cond = max(np.linalg.cond(np.eye(ni) - sv[:, None] * p * sv[None, :]) for p in P[q])
        assert cond < 100
        assert np.abs(W[q].cpu().numpy() - ref).max() < ni * cond * 2.0 ** -44 * np.abs(ref).max()
    ctx.close()


@pytest.mark.parametrize("ni,j", [(32, 5), (96, 40), (96, 70), (160, 159)])
def test_zero_pivot_is_reported(ni, j):
    """Pi_jj = 1 alone (v = 4, P_jj = 1/4: exact products) leaves a zero at elimination step j: info = j + 1
    for that system only."""
    torch, gw, cr, ctx = _ctx(ni, 1, 8, v=4.0)
    P = np.zeros((1, 8, ni, ni), complex)
    P[0, 3, j, j] = 0.25
    W = torch.zeros(1, 8, ni, ni, dtype=torch.complex128, device="cuda")
    info = torch.full((1, 8), -7, dtype=torch.int32, device="cuda")
    ctx.screen(0, 1, torch.from_numpy(P).cuda(), W, info, gw.GW_F32X2)
    ctx.sync()
    want = np.zeros((1, 8), np.int32)
    want[0, 3] = j + 1
    assert np.array_equal(info.cpu().numpy(), want)
    ctx.close()
