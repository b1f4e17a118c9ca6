"""The bosonic transforms on the tensor cores (GW_F32X2, csrc/digit_bose.cu) against the same maps in
64-bit sums: data rows that end inside a tile, several transforms per call, more than 64 tau (a row read
in two rounds), matrices that are no multiple of the 32 x 32 block, several pieces. Each product of
scaled row and column loses at most 2^-49 of the row's largest contribution (7 digits, the levels above
the sixth dropped), over 2 n terms."""
import numpy as np
import pytest

import gwinputs as gi

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,nt,count", [(32, 8, 1), (7, 16, 3), (45, 24, 2), (64, 72, 2), (160, 16, 9), (1, 8, 1)])
def test_bose_digits(m, nt, count):
    import torch

    import paper_1602_02313_gb300 as gw
    from paper_1602_02313_gb300 import build as b
    b.build()
    gr = gi.make_grid(60.0, nt, nt, nt, ncont=8)
    cr = gi.make_crystal(3, 1, 1, 1, 32, 60.0, qlist=[0])
    ctx = gw.GW(gr, cr, M=torch.zeros(1, 1, 32, 1, 1, dtype=torch.complex128, device="cuda"))
    T = gw.transform_matrices(gr)
    rng = np.random.default_rng(m + nt)
    amp = np.exp(-3.0 * rng.random(nt) * np.arange(nt) / 8)[None, :, None, None]  # data over many powers of two
    x = (rng.standard_normal((count, nt, m, m)) + 1j * rng.standard_normal((count, nt, m, m))) * amp
    y = torch.full((count, nt, m, m), float("nan"), dtype=torch.complex128, device="cuda")
    # forward
    ctx.tau_to_freq_many(gw.GW_BOSE, gw.GW_TAU_TO_IW, count, m * m, torch.from_numpy(x).cuda(), y, gw.GW_F32X2)
    ctx.sync()
    got = y.cpu().numpy()
    A = T["B_fwd"]
    ref = np.einsum("ji,ziab->zjab", A, x)
    col = np.abs(A).max(0)
    big = 2 * (col[None, :, None, None] * np.abs(x)).max(1, keepdims=True)  # largest contribution of each row
    rel = (np.abs(A) / col[None, :]).max(1)[None, :, None, None]
    assert (np.abs(got - ref) <= 2 * nt * 2.0 ** -49 * big * rel).all()
    # backward
    y.fill_(float("nan"))
    ctx.tau_to_freq_many(gw.GW_BOSE, gw.GW_IW_TO_TAU, count, m, torch.from_numpy(x).cuda(), y, gw.GW_F32X2)
    ctx.sync()
    got = y.cpu().numpy()
    R, I = T["B_bwd_re"], T["B_bwd_im"]
    xt = np.swapaxes(x, 2, 3)
    g, h = 0.5 * (x + xt), -0.5j * (x - xt)
    ap = lambda v: np.einsum("ij,zjab->ziab", R, v.real) + np.einsum("ij,zjab->ziab", I, v.imag)  # noqa: E731
    ref = ap(g) + 1j * ap(h)
    B = np.maximum(np.abs(R), np.abs(I))
    col = B.max(0)
    amax = np.maximum(np.abs(x), np.abs(xt))
    big = 2 * (col[None, :, None, None] * amax).max(1, keepdims=True)
    rel = (B / col[None, :]).max(1)[None, :, None, None]
    assert (np.abs(got - ref) <= 4 * nt * 2.0 ** -49 * big * rel).all()
    assert np.array_equal(got, np.conj(np.swapaxes(got, 2, 3)))
    ctx.close()
