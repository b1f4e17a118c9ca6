"""GW_FP64 contractions on rows whose entries spread over many powers of two, large ones of one row meeting tiny ones
of the other. The digit products (the default) are accurate relative to the rows' largest entries: n 2^-50 max|x|
max|y| for a sum of n terms, the bound of include/gw.h; the CUDA-core kernels (GW_TUNE_FP64_FORM 1) relative to each
term: n 2^-52 sum |x y|. The reference's own FP64 rounding is within the second bound, which is added to the first."""
import numpy as np
import pytest

import gwinputs as gi
import oracle as orc

pytestmark = pytest.mark.gpu

NK, NB, NI, NT = 2, 6, 64, 8


def _spread(rng, kind, shape):
    """Powers of two for M[k][I][a][b]: 1 in one half of the pairs and 2^-60 in the other, the halves exchanged from
    row to row; or 2^-40 .. 2^40 at random."""
    if kind == "random":
        return 2.0 ** rng.integers(-40, 41, shape)
    I, a = np.arange(shape[1])[:, None, None], np.arange(shape[2])[:, None]
    return np.broadcast_to(np.where((I + a) % 2 == 0, 1.0, 2.0 ** -60), shape)


@pytest.fixture(params=["crossed", "random"])
def case(request):
    import torch

    import paper_1602_02313_gb300 as gw
    from paper_1602_02313_gb300 import build as b
    b.build()
    rng = np.random.default_rng(41)
    cr = gi.make_crystal(41, NK, NB, NB // 2, NI, 20.0, qlist=[1])
    gr = gi.make_grid(20.0, NT, NT, NT, ncont=16)
    cplx = lambda *s: rng.standard_normal(s) + 1j * rng.standard_normal(s)  # noqa: E731
    M = cplx(NK, NI, NB, NB) * _spread(rng, request.param, (NK, NI, NB, NB))
    ctx = gw.GW(gr, cr, M=torch.from_numpy(np.ascontiguousarray(M[None])).cuda())
    G, occ = orc.green_tau0(cr.eps, gr.tau, gr.beta)
    W = cplx(NT, NI, NI) * 2.0 ** rng.integers(-30, 31, (NT, NI, NI))
    W = np.ascontiguousarray(W + np.conj(np.swapaxes(W, 1, 2)))
    yield torch, gw, ctx, M, G, occ, W, cr.kmq[0]
    ctx.close()


def _flat(M, k):
    return M[k].reshape(NI, -1)


def test_polarization(case):
    torch, gw, ctx, M, G, occ, W, kmq = case
    ref = orc.polarization(M, G, kmq)
    n = 2 * NK * NB * NB
    terms = np.zeros((NT, NI, NI))  # sum |w| |a| |a'|
    xmax, ymax = np.zeros((NT, NI)), np.zeros(NI)
    for k in range(NK):
        A = np.abs(_flat(M, k))
        ymax = np.maximum(ymax, A.max(1))
        for i in range(NT):
            w = np.abs(np.outer(G[kmq[k], :, NT - 1 - i], G[k, :, i])).reshape(-1)
            terms[i] += (A * w) @ A.T / NK
            xmax[i] = np.maximum(xmax[i], (A * w).max(1))
    rows = np.sqrt(2.0) * xmax[:, :, None] * ymax[None, None, :] / NK  # |re| + |im| <= sqrt(2) |a|
    rows = np.maximum(rows, np.swapaxes(rows, 1, 2))
    for form in (0, 1):
        ctx.set_tuning(gw.GW_TUNE_FP64_FORM, form)
        P = torch.full((NT, NI, NI), float("nan"), dtype=torch.complex128, device="cuda")
        ctx.polarization(0, torch.from_numpy(G).cuda(), P, gw.GW_FP64)
        ctx.sync()
        tol = 2 * n * 2.0 ** -52 * terms + (0.0 if form else np.sqrt(2.0) * n * 2.0 ** -50 * rows)
        assert (np.abs(P.cpu().numpy() - ref) <= tol).all(), form
    with pytest.raises(gw.GwError, match="GW_EINVAL"):
        ctx.set_tuning(gw.GW_TUNE_FP64_FORM, 2)


def test_selfenergy(case):
    torch, gw, ctx, M, G, occ, W, kmq = case
    ref, _, _ = orc.selfenergy(M, G, W, np.ones(NI), kmq, occ)
    terms, rows = np.zeros_like(ref), np.zeros_like(ref)
    for k in range(NK):
        A = np.abs(_flat(M, k))
        for i in range(NT):
            g = np.abs(G[kmq[k], :, i])[:, None]
            wmax = np.triu(np.abs(W[i])).max(0)  # column J over I <= J
            t = (A * (np.abs(W[i]) @ A)).sum(0)
            r = 2 * np.sqrt(2.0) * (A * wmax[:, None]).sum(0) * A.max(0)  # 2 sum_J (|re| + |im|) x a row of Y
            terms[k, :, i] = (g * t.reshape(NB, NB)).sum(0) / NK
            rows[k, :, i] = (g * r.reshape(NB, NB)).sum(0) / NK
    for form in (0, 1):
        ctx.set_tuning(gw.GW_TUNE_FP64_FORM, form)
        S = torch.zeros(NK, NB, NT, dtype=torch.float64, device="cuda")
        ctx.selfenergy(0, torch.from_numpy(G).cuda(), None, torch.from_numpy(W).cuda(), S, None, gw.GW_FP64)
        ctx.sync()
        tol = 2 * (2 * NI + NB) * 2.0 ** -52 * terms + (0.0 if form else 2 * NI * 2.0 ** -50 * rows)
        assert (np.abs(S.cpu().numpy() - ref) <= tol).all(), form


def test_selfenergy_offdiag(case):
    torch, gw, ctx, M, G, occ, W, kmq = case
    v = np.array(ctx.cr.v[0])
    ref, refx = orc.offdiag.selfenergy_offdiag(M, G, W, v, kmq, occ)
    terms, rows = np.zeros(ref.shape), np.zeros(ref.shape)
    tx, rx = np.zeros(refx.shape), np.zeros(refx.shape)
    n1, n2 = 2 * NI, 2 * NI * NB
    for k in range(NK):
        A = np.abs(M[k])  # [I][j][n]
        amax = A.max((0, 1))  # row n of the second product
        for i in range(NT):
            g = np.abs(G[kmq[k], :, i])
            Z = np.einsum("j,IJ,Jjm->Ijm", g, np.abs(W[i]), A)
            dZ = n1 * np.einsum("j,I,jm->Ijm", g, np.abs(W[i]).max(1), A.max(0))  # bound of Z's rows / 2^-50
            terms[k, :, :, i] = np.einsum("Ijn,Ijm->nm", A, Z) / NK
            rows[k, :, :, i] = (np.einsum("Ijn,Ijm->nm", A, dZ) + n2 * np.outer(amax, (Z + 2.0 ** -50 * dZ).max((0, 1)))) / NK
        Z = np.einsum("j,I,Ijm->Ijm", occ[kmq[k]], v, A)
        tx[k] = np.einsum("Ijn,Ijm->nm", A, Z) / NK
        rx[k] = n2 * np.outer(amax, Z.max((0, 1))) / NK
    for form in (0, 1):
        ctx.set_tuning(gw.GW_TUNE_FP64_FORM, form)
        S = torch.zeros(NK, NB, NB, NT, dtype=torch.complex128, device="cuda")
        Sx = torch.zeros(NK, NB, NB, dtype=torch.complex128, device="cuda")
        ctx.selfenergy_offdiag(0, torch.from_numpy(G).cuda(), torch.from_numpy(occ).cuda(), torch.from_numpy(W).cuda(), S, Sx)
        ctx.sync()
        f = 0.0 if form else 2.0 * 2.0 ** -50  # both parts of complex entries: sqrt(2) each way
        n = 2 * (n1 + n2)
        assert (np.abs(S.cpu().numpy() - ref) <= n * 2.0 ** -52 * terms + f * rows).all(), form
        assert (np.abs(Sx.cpu().numpy() - refx) <= n * 2.0 ** -52 * tx + f * rx).all(), form
