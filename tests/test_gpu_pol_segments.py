"""K segments of the tensor-core polarization (csrc/pol_plan.h): no segment may be empty. A block runs its
units one after another, and a unit without chunks has no operand to wait for, so it would complete the block's
accumulator barrier a second time while the unit before it is still being read. Host: every plan, over all
sizes (tests/pol_plan_check.cpp). GPU: P at sizes whose chunks do not divide into the wanted segments."""
import os
import shutil
import subprocess

import numpy as np
import pytest

import gwinputs as gi
import oracle as orc

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_1602_02313_gb300", "csrc")
TOL_P = 2e-5  # the tensor-core polarization's bound, as in test_gpu_mixed.py


def test_no_segment_is_empty(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    exe = str(tmp_path / "pol_plan_check")
    subprocess.run([cxx, "-O2", "-std=c++17", "-I", CSRC, os.path.join(HERE, "pol_plan_check.cpp"), "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    print(r.stdout)
    assert r.returncode == 0, r.stdout
    assert " 0 with an empty or overlong segment" in r.stdout


# (Nk, Nb, NI, tau): on 152 SMs the wanted segments (10, 7, 13, 5) leave 8, 6, 12 and 4 of them with chunks
@pytest.mark.gpu
@pytest.mark.parametrize("nk,nb,ni,nt", [(4, 16, 64, 32), (3, 16, 64, 48), (8, 24, 96, 24), (2, 16, 288, 16)])
def test_polarization(nk, nb, ni, nt):
    import torch

    import paper_1602_02313_gb300 as gw
    from paper_1602_02313_gb300 import build as b
    b.build()
    cr = gi.make_crystal(ni + nt, nk, nb, nb // 2, ni, 40.0, qlist=[1])
    gr = gi.make_grid(40.0, nt, nt, nt, ncont=16)
    ctx = gw.GW(gr, cr, omega=1.0)
    G, _ = orc.green_tau0(cr.eps, gr.tau, gr.beta)
    ref = orc.polarization(gi.m_for_q(cr, 0), G, cr.kmq[0])
    P = torch.full((nt, ni, ni), float("nan"), dtype=torch.complex128, device="cuda")
    ctx.polarization(0, torch.from_numpy(G).cuda(), P, gw.GW_FP16X2)
    ctx.sync()
    assert np.abs(P.cpu().numpy() - ref).max() < TOL_P * np.abs(ref).max()
    ctx.close()
