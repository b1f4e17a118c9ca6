"""gw_dyson_matrix at the sizes where its elimination changes: one band, one full warp of columns and one more, and
the last size whose matrix is in shared memory (113) beside the first that is in the workspace; Hermitian parts that
force row exchanges (their diagonal is zero but for the band energies). Against the oracle's solve in i w. Tolerance:
elimination nb eps cond, cond below |H| / (pi T) ~ 200, times the maps' gain (< 100): 114 x 200 x 100 x 2^-53 = 3e-10."""
import numpy as np
import pytest

import gwinputs as gi
import oracle as orc
from oracle import offdiag as od

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nb", [1, 2, 32, 33, 113, 114])
def test_dyson_matrix_sizes(nb):
    import torch

    import paper_1602_02313_gb300 as gw
    from paper_1602_02313_gb300 import build as b
    b.build()
    cr = gi.make_crystal(nb, 2, nb, max(1, nb // 2), 32, 40.0, qlist=[1])
    gr = gi.make_grid(40.0, 16, 16, 16, ncont=16)
    ctx = gw.GW(gr, cr, M=torch.zeros(1, 2, 32, nb, nb, dtype=torch.complex128, device="cuda"))
    rng = np.random.default_rng(nb)
    X = rng.standard_normal((2, nb, nb)) + 1j * rng.standard_normal((2, nb, nb))
    Sx = 0.5 * (X + np.conj(np.swapaxes(X, 1, 2)))
    Sx[:, np.arange(nb), np.arange(nb)] = 0.0
    g0, _ = orc.green_tau0(rng.uniform(-1.5, 1.5, (1, 3)), gr.tau, gr.beta)
    C = 0.2 * (rng.standard_normal((2, nb, 3)) + 1j * rng.standard_normal((2, nb, 3)))
    Sc = np.einsum("knp,pt,kmp->knmt", C, g0[0], np.conj(C))
    d = lambda x: torch.from_numpy(np.ascontiguousarray(x)).cuda()
    G = torch.zeros(2, nb, nb, 16, dtype=torch.complex128, device="cuda")
    occ = torch.zeros(2, nb, nb, dtype=torch.complex128, device="cuda")
    info = torch.full((2,), -1, dtype=torch.int32, device="cuda")
    ctx.dyson_matrix(d(cr.eps), d(Sx), None, d(Sc), G, occ, info)
    ctx.sync()
    Gr, occr = od.dyson_matrix_iw(cr.eps, Sx, 0.0 * Sx, orc.sigma_tau_to_iw(Sc, gr), gr)
    assert int(info.max()) < 2  # no zero pivot (1: the eigensolver stopped above 1e-15, G is written)
    assert np.abs(G.cpu().numpy() - Gr).max() < 3e-10 * np.abs(Gr).max()
    assert np.abs(occ.cpu().numpy() - occr).max() < 3e-10 * np.abs(occr).max()
    ctx.close()
