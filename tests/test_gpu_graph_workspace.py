"""A captured call keeps the workspace it was captured with: a larger call afterwards gets a new one, and the
graph replays to the same bits. Each case warms the small call up, captures it, runs a call that needs more
workspace, and replays."""
import numpy as np
import pytest

import gwinputs as gi

pytestmark = pytest.mark.gpu

NI, NT = 64, 8


def _c(rng, *s):
    import torch
    x = rng.standard_normal(s + (2,))
    return torch.from_numpy(np.ascontiguousarray(x)).cuda().view(torch.complex128)[..., 0].contiguous()


def _cases(gw, ctx, rng, torch):
    """name: (small call, larger call, outputs of the small one)"""
    z = lambda *s, dt=torch.complex128: torch.zeros(s, dtype=dt, device="cuda")  # noqa: E731
    nq, nk, nb = ctx.cr.nq, ctx.cr.nk, ctx.cr.nb
    Pt, Wv = _c(rng, nq, NT, NI, NI), _c(rng, nq, NT, NI, NI)
    X = 0.01 * _c(rng, nq, NT, NI, NI)
    Pv = -(X @ X.mH)
    G = torch.from_numpy(-rng.uniform(0.1, 1.0, (nk, nb, NT))).cuda()
    occ = torch.from_numpy(rng.uniform(0.0, 1.0, (nk, nb))).cuda()
    H = X[0] + X[0].mH
    big, info = z(nq, NT, NI, NI), z(nq, NT, dt=torch.int32)
    fwd, bwd, scr = z(1, NT, NI, NI), z(1, NT, NI, NI), z(1, NT, NI, NI)
    S, Sb, Sx = z(nk, nb, nb, NT), z(nk, nb, nb, NT), z(nk, nb, nb)
    eps = torch.from_numpy(ctx.cr.eps).cuda()
    G1, occ1, G2 = z(nk, nb, nb, NT), z(nk, nb, nb), z(nk, nb, nb, NT)
    vx, dinfo = z(nk, nb, nb), z(nk, dt=torch.int32)
    F, R = gw.GW_TAU_TO_IW, gw.GW_IW_TO_TAU
    many = lambda d, n, b, i, o: ctx.tau_to_freq_many(gw.GW_BOSE, d, n, b, i, o, gw.GW_F32X2)  # noqa: E731
    return {
        "forward": (lambda: many(F, 1, NI * NI, Pt, fwd), lambda: many(F, nq, NI * NI, Pt, big), [fwd]),
        "backward": (lambda: many(R, 1, NI, Wv, bwd), lambda: many(R, nq, NI, Wv, big), [bwd]),
        "screen": (lambda: ctx.screen(0, 1, Pv, scr, info, gw.GW_F32X2),
                   lambda: ctx.screen(0, nq, Pv, big, info, gw.GW_F32X2), [scr]),
        "offdiag": (lambda: (S.zero_(), ctx.selfenergy_offdiag(0, G, occ, H, S, None)),
                    lambda: ctx.selfenergy_offdiag(0, G, occ, H, Sb, Sx), [S]),
        "dyson_matrix": (lambda: ctx.dyson_matrix(eps, vx, vx, None, G1, occ1, dinfo),
                         lambda: ctx.dyson_matrix(eps, vx, vx, Sb, G2, occ1, dinfo), [G1]),
    }


@pytest.mark.parametrize("name", ["forward", "backward", "screen", "offdiag", "dyson_matrix"])
def test_replay_after_a_larger_call(name):
    import torch

    import paper_1602_02313_gb300 as gw
    from paper_1602_02313_gb300 import build as b
    b.build()
    rng = np.random.default_rng(17)
    cr = gi.make_crystal(5, 4, 8, 4, NI, 30.0, qlist=[1, 2, 3, 0])
    gr = gi.make_grid(30.0, NT, NT, NT, ncont=16)
    ctx = gw.GW(gr, cr, M=_c(rng, 4, 4, NI, 8, 8))
    small, large, out = _cases(gw, ctx, rng, torch)[name]
    st = torch.cuda.Stream()
    st.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(st):
        ctx.set_stream(st)
        small()
        st.synchronize()
        ref = [o.clone() for o in out]
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=st):
            small()
        large()
        st.synchronize()
        for o in out:
            o.fill_(float("nan"))
        g.replay()
        st.synchronize()
        assert all(bool(torch.isfinite(torch.view_as_real(r)).all()) and torch.equal(o, r) for o, r in zip(out, ref))
        ctx.sync()
    ctx.close()


def test_seed_network_replay_after_a_larger_batch():
    import torch

    import paper_1602_02313_gb300 as gw
    from paper_1602_02313_gb300 import build as b
    b.build()
    rng = np.random.default_rng(18)
    x = torch.from_numpy(rng.standard_normal((1024, 64)).astype(np.float32)).cuda()
    A = torch.from_numpy((0.1 * rng.standard_normal((64, 128))).astype(np.float32)).cuda()
    st = torch.cuda.Stream()
    st.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(st):
        net = gw.MLP(nin=64, nh=128, nhidden=2, nout=128, seed=2, stream=st)
        loss = torch.zeros(1, dtype=torch.float32, device="cuda")
        g1, g2 = (torch.zeros(net.num_params(), dtype=torch.float32, device="cuda") for _ in range(2))
        net.loss_grad(x[:128], A, loss, g1)
        st.synchronize()
        ref = g1.clone()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=st):
            net.loss_grad(x[:128], A, loss, g1)
        net.loss_grad(x, A, loss, g2)
        st.synchronize()
        g1.fill_(float("nan"))
        graph.replay()
        st.synchronize()
        assert bool(torch.isfinite(ref).all()) and torch.equal(g1, ref)
        net.sync()
    net.close()


def test_continuation_replay_after_another_grid():
    """A captured continuation keeps its pole grid: another gw_cpe_setup and a larger fit after it, then the replay."""
    import torch

    import paper_1602_02313_gb300 as gw
    from paper_1602_02313_gb300 import build as b
    from paper_1602_02313_gb300.driver import cpe_grid
    b.build()
    rng = np.random.default_rng(19)
    cr = gi.make_crystal(6, 4, 8, 4, NI, 30.0, qlist=[1])
    gr = gi.make_grid(30.0, NT, NT, NT, ncont=64)
    st = torch.cuda.Stream()
    ctx = gw.GW(gr, cr, M=_c(rng, 1, 4, NI, 8, 8), stream=st)
    n = 32
    w = (2 * np.arange(64) + 1) * np.pi / 30.0
    pole, res = rng.uniform(-1.0, 1.0, (2 * n, 3)), rng.uniform(0.05, 0.2, (2 * n, 3))
    sig = torch.from_numpy((res[:, :, None] / (1j * w - pole[:, :, None])).sum(1)).cuda()
    d = {k: torch.from_numpy(rng.uniform(-0.5, 0.5, 2 * n)).cuda() for k in ("eps", "sigx", "vxc")}
    eqp, info = torch.zeros(2 * n, dtype=torch.float64, device="cuda"), torch.zeros(2 * n, dtype=torch.int32, device="cuda")
    x = cpe_grid()
    torch.cuda.synchronize()

    def fit(m):
        ctx.continue_(gw.GW_CPE, sig[:m], d["eps"][:m], d["sigx"][:m], d["vxc"][:m], None, None, eqp[:m], info[:m])

    with torch.cuda.stream(st):
        ctx.cpe_setup(x, 1e-3)
        fit(n)
        st.synchronize()
        ref = eqp[:n].clone()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=st):
            fit(n)
        ctx.cpe_setup(x[::2].copy(), 1e-4)
        fit(2 * n)
        st.synchronize()
        eqp.fill_(float("nan"))
        g.replay()
        st.synchronize()
        assert bool(torch.isfinite(ref).all()) and torch.equal(eqp[:n], ref)
        ctx.sync()
    ctx.close()
