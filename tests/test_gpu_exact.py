"""The FP64 contractions on the tensor cores (exact digit products, csrc/exact_tc.cu).

Against plain FP64 sums at the edges of the tiles: bases that fill half a 64-column tile or a
128-row tile, band counts whose pairs end inside an 8-pair chunk or a 128-row tile, one K block
and many. The tolerance is the FP64 rounding bound of the reference sum itself, n 2^-53 sum |a||b|
with n the number of terms; the digit sums lose 2^-52 max|a| max|b| per term.
"""
import numpy as np
import pytest

import gwinputs as gi
import oracle as orc

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gw():
    from paper_1602_02313_gb300 import build as b
    b.build()
    import paper_1602_02313_gb300 as pkg
    return pkg


def _setup(gw, nk, nb, ni, nt, seed, rows=None):
    import torch
    rng = np.random.default_rng(seed)
    cr = gi.make_crystal(seed, nk, nb, max(1, nb // 2), ni, 30.0, qlist=[1 % nk])
    gr = gi.make_grid(30.0, nt, nt, nt, ncont=16)
    M = (rng.standard_normal((nk, ni, nb, nb)) + 1j * rng.standard_normal((nk, ni, nb, nb))) * np.sqrt(0.5 / nb)
    if rows is not None:
        M *= rows[None, :, None, None]
    ctx = gw.GW(gr, cr, M=torch.from_numpy(np.ascontiguousarray(M[None])).cuda())
    G, occ = orc.green_tau0(cr.eps, gr.tau, gr.beta)
    return torch, rng, cr, gr, M, ctx, G, occ


def _pol(torch, gw, ctx, G, nt, ni):
    P = torch.full((nt, ni, ni), float("nan"), dtype=torch.complex128, device="cuda")
    ctx.polarization(0, torch.from_numpy(G).cuda(), P, gw.GW_FP64)
    ctx.sync()
    return P.cpu().numpy()


def _pol_scale(M, G, kmq):
    """sum |w| |a| |a'| of every element: the FP64 rounding bound's sum."""
    nt = G.shape[-1]
    out = np.zeros((nt, M.shape[1], M.shape[1]))
    for k in range(M.shape[0]):
        A = np.abs(M[k]).reshape(M.shape[1], -1)
        for i in range(nt):
            w = np.abs(np.outer(G[kmq[k], :, nt - 1 - i], G[k, :, i])).reshape(-1)
            out[i] += (A * w) @ A.T
    return out / M.shape[0]


SHAPES = [(2, 4, 32, 8), (1, 3, 64, 8), (3, 5, 96, 8), (2, 12, 160, 8), (2, 8, 288, 8), (5, 16, 64, 24)]


@pytest.mark.parametrize("nk,nb,ni,nt", SHAPES)
def test_polarization(gw, nk, nb, ni, nt):
    torch, rng, cr, gr, M, ctx, G, occ = _setup(gw, nk, nb, ni, nt, 300 + ni)
    got = _pol(torch, gw, ctx, G, nt, ni)
    ref = orc.polarization(M, G, cr.kmq[0])
    n = 4 * nk * nb * nb
    assert (np.abs(got - ref) <= n * 2.0 ** -52 * _pol_scale(M, G, cr.kmq[0])).all()
    assert np.array_equal(got, np.conj(np.swapaxes(got, 1, 2)))  # exactly Hermitian
    ctx.close()


def test_polarization_rows_of_any_size(gw):
    """Rows scaled by 2^-400 .. 2^400, a zero row and a row that is not finite: each element is accurate
    relative to its own rows, and only the rows and columns that are not finite are nan."""
    ni = 64
    rows = np.ones(ni)
    rows[:8] = 2.0 ** np.array([-400, -90, -30, -3, 3, 30, 90, 400])
    rows[9] = 0.0
    torch, rng, cr, gr, M, ctx, G, occ = _setup(gw, 2, 6, ni, 8, 77, rows)
    ref = orc.polarization(M, G, cr.kmq[0])
    bound = 4 * 2 * 36 * 2.0 ** -52 * _pol_scale(M, G, cr.kmq[0])
    assert (np.abs(_pol(torch, gw, ctx, G, 8, ni) - ref) <= bound).all()
    ctx._M[0, 0, 10, 1, 2] = float("inf")
    got = _pol(torch, gw, ctx, G, 8, ni)
    ok = np.arange(ni) != 10
    assert np.isnan(got[:, 10, :]).all() and np.isnan(got[:, :, 10]).all()
    assert (np.abs(got - ref)[:, ok][:, :, ok] <= bound[:, ok][:, :, ok]).all()
    ctx.close()


@pytest.mark.parametrize("nk,nb,ni,nt", SHAPES)
def test_selfenergy(gw, nk, nb, ni, nt):
    torch, rng, cr, gr, M, ctx, G, occ = _setup(gw, nk, nb, ni, nt, 500 + ni)
    X = rng.standard_normal((nt, ni, ni)) + 1j * rng.standard_normal((nt, ni, ni))
    W = X + np.conj(np.swapaxes(X, 1, 2))
    W = np.ascontiguousarray(W + 1e-3 * X)  # not Hermitian: the result is the real part, which sees the Hermitian part only
    S = torch.from_numpy(np.full((nk, nb, nt), 0.25)).cuda()  # accumulated into
    ctx.selfenergy(0, torch.from_numpy(G).cuda(), None, torch.from_numpy(W).cuda(), S, None, gw.GW_FP64)
    ctx.sync()
    ref, _, _ = orc.selfenergy(M, G, W, cr.v[0], cr.kmq[0], occ)
    scale = np.zeros_like(ref)
    for k in range(nk):
        A = np.abs(M[k]).reshape(ni, -1)
        for i in range(nt):
            d = (A * (np.abs(W[i]) @ A)).sum(0).reshape(nb, nb)
            scale[k, :, i] = (np.abs(G[cr.kmq[0][k], :, i])[:, None] * d).sum(0) / nk
    assert (np.abs(S.cpu().numpy() - 0.25 - ref) <= (2 * ni + nb) * 2.0 ** -52 * scale + 2.0 ** -54).all()
    ctx.close()


def test_captured_without_workspace(gw):
    """A first call under stream capture cannot allocate the digit workspace: the kernels that need none run,
    with the same values to FP64 rounding."""
    import torch as _t
    torch, rng, cr, gr, M, ctx, G, occ = _setup(gw, 2, 4, 64, 8, 9)
    Gd = torch.from_numpy(G).cuda()
    P = torch.zeros(8, 64, 64, dtype=torch.complex128, device="cuda")
    W = torch.from_numpy(rng.standard_normal((8, 64, 64)) + 0j).cuda()
    W = W + W.mH
    S = torch.zeros(2, 4, 8, dtype=torch.float64, device="cuda")
    g = _t.cuda.CUDAGraph()
    with _t.cuda.graph(g):
        ctx.set_stream(_t.cuda.current_stream())
        ctx.polarization(0, Gd, P, gw.GW_FP64)
        ctx.selfenergy(0, Gd, None, W, S, None, gw.GW_FP64)
    g.replay()
    _t.cuda.synchronize()
    ctx.set_stream(_t.cuda.current_stream())
    P1, S1 = torch.zeros_like(P), torch.zeros_like(S)
    ctx.polarization(0, Gd, P1, gw.GW_FP64)
    ctx.selfenergy(0, Gd, None, W, S1, None, gw.GW_FP64)
    ctx.sync()
    assert float((P - P1).abs().max()) <= 128 * 2.0 ** -52 * float(P1.abs().max())
    assert float((S - S1).abs().max()) <= 128 * 2.0 ** -52 * float(S1.abs().max())
    ctx.close()


def test_stalled_pipeline_reports_and_recovers(gw):
    """The digit GEMM's waits are bounded like the mixed kernels': an injected stall (1 ms budget) is reported by
    gw_sync, and the same context then gives the healthy values again, bit for bit."""
    torch, rng, cr, gr, M, ctx, G, occ = _setup(gw, 2, 6, 96, 8, 12)
    X = rng.standard_normal((8, 96, 96))
    W = torch.from_numpy(np.ascontiguousarray(X + np.swapaxes(X, 1, 2)) + 0j).cuda()
    Gd = torch.from_numpy(G).cuda()

    def run():
        P = torch.zeros(8, 96, 96, dtype=torch.complex128, device="cuda")
        S = torch.zeros(2, 6, 8, dtype=torch.float64, device="cuda")
        ctx.polarization(0, Gd, P, gw.GW_FP64)
        ctx.selfenergy(0, Gd, None, W, S, None, gw.GW_FP64)
        return P, S

    P0, S0 = run()
    ctx.sync()
    ctx.set_tuning(gw.GW_TUNE_WAIT_CYCLES, 2_000_000)
    ctx.set_tuning(gw.GW_TUNE_FAULT_STALL, 1)
    run()
    with pytest.raises(gw.GwError, match="GW_ETIMEOUT"):
        ctx.sync()
    ctx.set_tuning(gw.GW_TUNE_FAULT_STALL, 0)
    ctx.set_tuning(gw.GW_TUNE_WAIT_CYCLES, 4_000_000_000)
    P1, S1 = run()
    ctx.sync()
    assert torch.equal(P0, P1) and torch.equal(S0, S1)
    ctx.close()
