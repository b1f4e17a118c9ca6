"""What a context keeps on the device between calls (the staged operands of one q, the matrix elements of one q) is
what the last executed call left there, and a captured call executes when its graph is replayed: a graph has to bring
its own, and an eager call after a capture must not take the captured call's for done."""
import numpy as np
import pytest

import gwinputs as gi
import oracle as orc

pytestmark = pytest.mark.gpu

NT = 8


def _setup(m_mode):
    import torch

    import paper_1602_02313_gb300 as gw
    from paper_1602_02313_gb300 import build as b
    b.build()
    cr = gi.make_crystal(31, 3, 6, 3, 64, 30.0, qlist=[0, 1])
    gr = gi.make_grid(30.0, NT, NT, NT, ncont=16)
    st = torch.cuda.Stream()
    ctx = gw.GW(gr, cr, stream=st, m_mode=m_mode)
    G, occ = orc.green_tau0(cr.eps, gr.tau, gr.beta)
    st.wait_stream(torch.cuda.current_stream())
    return torch, gw, st, ctx, torch.from_numpy(G).cuda(), torch.from_numpy(occ).cuda()


def _capture(torch, st, call):
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=st):
        call()
    return g


def _check(torch, st, ctx, call, out):
    """call(q) writes out; q = 0 and 1 eagerly, then around captures."""
    def eager(q):
        out.fill_(float("nan"))
        call(q)
        st.synchronize()
        return out.clone()

    def replay(g):
        out.fill_(float("nan"))
        g.replay()
        st.synchronize()
        return out.clone()

    with torch.cuda.stream(st):
        ref = [eager(0), eager(1)]
        assert not torch.equal(ref[0], ref[1]) and bool(torch.isfinite(torch.view_as_real(ref[0] + 0j)).all())
        g1 = _capture(torch, st, lambda: call(1))  # captured with q = 1 staged
        assert torch.equal(eager(0), ref[0])
        assert torch.equal(replay(g1), ref[1])     # replayed with q = 0 staged
        assert torch.equal(eager(0), ref[0])
        g1 = _capture(torch, st, lambda: call(1))  # captured with q = 0 staged, not replayed
        assert torch.equal(eager(1), ref[1])
        assert torch.equal(eager(0), ref[0])
        assert torch.equal(replay(g1), ref[1])
        assert torch.equal(eager(0), ref[0])       # q = 0 was staged before the replay
        ctx.sync()
    ctx.close()


@pytest.mark.parametrize("m_mode", [1, 2])
def test_selfenergy(m_mode):
    torch, gw, st, ctx, G, occ = _setup(m_mode)
    rng = np.random.default_rng(4)
    X = rng.standard_normal((NT, 64, 64)) + 1j * rng.standard_normal((NT, 64, 64))
    W = torch.from_numpy(np.ascontiguousarray(X + np.conj(np.swapaxes(X, 1, 2)))).cuda()
    S = torch.zeros(3, 6, NT, dtype=torch.float64, device="cuda")

    def call(q):
        S.zero_()
        ctx.selfenergy(q, G, occ, W, S, None, gw.GW_FP16X2)

    torch.cuda.synchronize()
    _check(torch, st, ctx, call, S)


@pytest.mark.parametrize("prec", ["fp64", "fp16x2"])
def test_polarization_with_generated_elements(prec):
    torch, gw, st, ctx, G, occ = _setup(2)
    P = torch.zeros(NT, 64, 64, dtype=torch.complex128, device="cuda")
    torch.cuda.synchronize()
    _check(torch, st, ctx, lambda q: ctx.polarization(q, G, P, gw.PREC[prec]), P)


@pytest.mark.parametrize("first,second", [(1, 2), (2, 1)])
def test_polarization_forms(first, second):
    """A graph of one form of P replays to the same bits after eager calls of the other, whose strips differ."""
    import torch

    import paper_1602_02313_gb300 as gw
    from paper_1602_02313_gb300 import build as b
    b.build()
    cr = gi.make_crystal(32, 2, 8, 4, 160, 30.0, qlist=[1])
    gr = gi.make_grid(30.0, NT, NT, NT, ncont=16)
    G, _ = orc.green_tau0(cr.eps, gr.tau, gr.beta)
    Gd = torch.from_numpy(G).cuda()
    P = torch.zeros(NT, 160, 160, dtype=torch.complex128, device="cuda")
    st = torch.cuda.Stream()
    ctx = gw.GW(gr, cr, stream=st, m_mode=1)
    torch.cuda.synchronize()
    with torch.cuda.stream(st):
        ref = {}
        for form in (first, second, first):
            ctx.set_tuning(gw.GW_TUNE_POL_FORM, form)
            ctx.polarization(0, Gd, P, gw.GW_FP16X2)
            st.synchronize()
            assert form not in ref or torch.equal(ref[form], P)
            ref[form] = P.clone()
        assert not torch.equal(ref[first], ref[second])
        g = _capture(torch, st, lambda: ctx.polarization(0, Gd, P, gw.GW_FP16X2))
        for form in (second, first):
            ctx.set_tuning(gw.GW_TUNE_POL_FORM, form)
            ctx.polarization(0, Gd, P, gw.GW_FP16X2)
            st.synchronize()
            assert torch.equal(P, ref[form])
            P.fill_(float("nan"))
            g.replay()
            st.synchronize()
            assert torch.equal(P, ref[first])
        ctx.sync()
    ctx.close()
