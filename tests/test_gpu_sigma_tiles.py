"""Tensor-core self-energy at the edges of its column parts and K steps: one 32-column chunk, an odd
number of 16-column blocks per half, and bases above 256 whose parts end inside a 32-wide chunk (NI =
288, 352, 416), against the FP64 self-energy, within the tensor-core bound 2e-5 of the largest value."""
import numpy as np
import pytest

import gwinputs as gi
import oracle as orc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ni", [32, 96, 160, 256, 288, 352, 416, 512])
def test_selfenergy_mixed(ni):
    import torch

    import paper_1602_02313_gb300 as gw
    from paper_1602_02313_gb300 import build as b
    b.build()
    nk, nb, nt = 2, 7, 8
    rng = np.random.default_rng(ni)
    cr = gi.make_crystal(ni, nk, nb, 3, ni, 30.0, qlist=[1])
    gr = gi.make_grid(30.0, nt, nt, nt, ncont=16)
    M = (rng.standard_normal((1, nk, ni, nb, nb)) + 1j * rng.standard_normal((1, nk, ni, nb, nb))) * np.sqrt(0.5 / nb)
    ctx = gw.GW(gr, cr, M=torch.from_numpy(M).cuda())
    G, occ = (torch.from_numpy(x).cuda() for x in orc.green_tau0(cr.eps, gr.tau, gr.beta))
    X = rng.standard_normal((nt, ni, ni)) + 1j * rng.standard_normal((nt, ni, ni))
    W = torch.from_numpy(np.ascontiguousarray(X @ np.conj(np.swapaxes(X, 1, 2)) / ni)).cuda()
    out = []
    for prec in (gw.GW_FP64, gw.GW_FP16X2):
        S = torch.zeros(nk, nb, nt, dtype=torch.float64, device="cuda")
        ctx.selfenergy(0, G, occ, W, S, None, prec)
        ctx.sync()  # also reports a pipeline wait that ran out
        out.append(S)
    assert float((out[0] - out[1]).abs().max()) < 2e-5 * float(out[0].abs().max())
    ctx.close()
