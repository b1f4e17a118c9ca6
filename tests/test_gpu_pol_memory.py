"""The tensor-core polarization where memory is short: fewer K segments of partials per pass, then the form of P that
needs no FP32 image of the matrix elements; GW_ENOMEM only when not even that fits. The rest of the memory is held by a
tensor that nothing touches."""
import numpy as np
import pytest

import gwinputs as gi
import oracle as orc

pytestmark = pytest.mark.gpu

TOL_P = 2e-5  # the tensor-core polarization's bound, as in test_gpu_mixed.py
MIB = 1 << 20
# Nk 16, Nb 64, NI 256, 16 tau: operand image 128 MiB, its FP32 image another 128, weights 4, E 8 MiB, and for each of 64
# segments partials of 4 MiB (E form) or 8 (the other form): 524 MiB, 272 with one segment per pass; 140 in the other form
NK, NB, NI, NT = 16, 64, 256, 16


@pytest.mark.parametrize("left_mib,form", [(2048, 1), (420, 1), (230, 1)])
def test_polarization(left_mib, form):
    import torch

    import paper_1602_02313_gb300 as gw
    from paper_1602_02313_gb300 import build as b
    b.build()
    cr = gi.make_crystal(23, NK, NB, NB // 2, NI, 40.0, qlist=[1])
    gr = gi.make_grid(40.0, NT, NT, NT, ncont=16)
    torch.manual_seed(5)
    M = torch.randn(1, NK, NI, NB, NB, dtype=torch.complex128, device="cuda") * NB ** -0.5
    G, _ = orc.green_tau0(cr.eps, gr.tau, gr.beta)
    Gd = torch.from_numpy(G).cuda()
    P = [torch.zeros(NT, NI, NI, dtype=torch.complex128, device="cuda") for _ in range(3)]
    ctx = gw.GW(gr, cr, M=M)
    ctx.set_tuning(gw.GW_TUNE_POL_FORM, form)
    ctx.polarization(0, Gd, P[0], gw.GW_FP16X2)  # plenty of memory: the reference bits of this form
    ctx.sync()
    ctx.close()
    ctx = gw.GW(gr, cr, M=M)
    torch.cuda.synchronize()
    hold = []  # down to left_mib, in pieces as large as can be had
    while (n := torch.cuda.mem_get_info()[0] // MIB - left_mib) > 0:
        for part in (n, n // 2, n // 8, 2):
            try:
                hold.append(torch.empty(part * MIB, dtype=torch.uint8, device="cuda"))
                break
            except torch.OutOfMemoryError:
                assert part > 2
        else:
            break
    try:
        ctx.polarization(0, Gd, P[1], gw.GW_FP16X2)
        ctx.polarization(0, Gd, P[2], gw.GW_FP16X2)
        ctx.sync()
    finally:
        del hold
        torch.cuda.empty_cache()
    assert torch.equal(P[1], P[2])
    scale = P[0].abs().max()
    assert (P[1] - P[0]).abs().max() < TOL_P * scale
    ctx.close()
