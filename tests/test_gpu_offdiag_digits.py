"""gw_selfenergy_offdiag by digit products (csrc/digit_offdiag.cu) against complex128 sums of the same terms, W~ not
Hermitian, and its CUDA-core form (what a first call under capture runs): rows that end inside a tile, several tiles of
columns, and sizes whose k points and tau go in groups. Tolerance per element, relative to the sum of the terms'
magnitudes: two operands cut at 2^-56 of their row's largest value over nb ni terms, and 2e-14 for the FP64 sums."""
import numpy as np
import pytest

import gwinputs as gi
import oracle as orc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nk,nb,ni,ntau,exchange,capture", [
    (2, 3, 32, 8, True, False), (3, 5, 96, 12, False, False), (2, 33, 64, 8, True, False), (3, 16, 32, 8, True, True),
    (4, 48, 256, 32, True, False), (1, 64, 384, 32, True, False)])
def test_offdiag_digits(nk, nb, ni, ntau, exchange, capture):
    import torch

    import paper_1602_02313_gb300 as gw
    from paper_1602_02313_gb300 import build as b
    b.build()
    cr = gi.make_crystal(7, nk, nb, max(1, nb // 2), ni, 60.0, qlist=[nk - 1])
    gr = gi.make_grid(60.0, ntau, ntau, ntau, ncont=8)
    M = torch.from_numpy(np.ascontiguousarray(gi.m_for_q(cr, 0))).cuda().reshape(nk, ni, nb, nb)
    ctx = gw.GW(gr, cr, omega=1.3, M=M.reshape(1, nk, ni, nb, nb))
    Gh, occh = orc.green_tau0(cr.eps, gr.tau, gr.beta)
    G, occ = torch.from_numpy(Gh).cuda(), torch.from_numpy(occh).cuda()
    c16 = dict(dtype=torch.complex128, device="cuda")
    torch.manual_seed(ni + nb)
    W = torch.randn(ntau, ni, ni, **c16)
    S, Sx = torch.ones(nk, nb, nb, ntau, **c16), torch.ones(nk, nb, nb, **c16)
    torch.cuda.synchronize()
    if capture:
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            ctx.set_stream(torch.cuda.current_stream())
            ctx.selfenergy_offdiag(0, G, occ, W, S, Sx if exchange else None)
        g.replay()
        torch.cuda.synchronize()
        ctx.set_stream(torch.cuda.current_stream())
    else:
        ctx.selfenergy_offdiag(0, G, occ, W, S, Sx if exchange else None)
    ctx.sync()
    torch.cuda.synchronize()
    v, tol = torch.from_numpy(np.ascontiguousarray(cr.v[0])).cuda(), nb * ni * 2.0**-54 + 2e-14
    pref = -1.0 / (1.3 * nk)
    for k in range(nk):
        a, km = M[k], int(cr.kmq[0][k])
        x, y = a.permute(1, 0, 2).reshape(nb * ni, nb), a.reshape(ni, nb * nb)
        for t in range(0, ntau, 5):
            Z = ((W[t] @ y).reshape(ni, nb, nb) * G[km, :, t].reshape(1, nb, 1)).permute(1, 0, 2).reshape(nb * ni, nb)
            m = ((W[t].abs() @ y.abs()).reshape(ni, nb, nb) * G[km, :, t].abs().reshape(1, nb, 1)).permute(1, 0, 2)
            mag = abs(pref) * (x.abs().T @ m.reshape(nb * ni, nb)) + 1.0
            assert ((S[k, :, :, t] - 1.0 - pref * (x.conj().T @ Z)).abs() / mag).max().item() < tol
        if exchange:
            f = (occ[km].reshape(nb, 1, 1) * v.reshape(1, ni, 1)).expand(nb, ni, nb).reshape(nb * ni, nb)
            mag = abs(pref) * (x.abs().T @ (f * x).abs()) + 1.0
            assert ((Sx[k] - 1.0 - pref * (x.conj().T @ (f * x))).abs() / mag).max().item() < tol
    if not exchange:
        assert bool((Sx == 1.0).all())
    ctx.close()
