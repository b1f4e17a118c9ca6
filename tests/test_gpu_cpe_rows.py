"""The CPE fit's two launches: with more problems than fit resident the factor keeps 64 rows at first, and a passive
set that outgrows them (a seed on the whole grid) is done again with all rows. A batch gives, bit for bit, what its
problems give one by one (one launch with all rows)."""
import numpy as np
import pytest

import gwinputs as gi

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("seeded", [False, True])
def test_batch_equals_single(seeded):
    import torch

    import paper_1602_02313_gb300 as gw
    from paper_1602_02313_gb300 import build as b
    from paper_1602_02313_gb300.driver import cpe_grid
    b.build()
    nk, nb, nc = 170, 4, 32
    cr = gi.make_crystal(3, nk, nb, 2, 32, 40.0, qlist=[0])
    gr = gi.make_grid(40.0, 16, 16, 16, ncont=nc)
    ctx = gw.GW(gr, cr, M=torch.zeros(1, nk, 32, nb, nb, dtype=torch.complex128, device="cuda"))
    ctx.cpe_setup(cpe_grid(), 1e-3)
    n = nk * nb
    rng = np.random.default_rng(4)
    w = (2 * np.arange(nc) + 1) * np.pi / 40.0
    E, A = rng.uniform(-2, 2, (n, 6)), rng.uniform(0.1, 1.0, (n, 6))
    S = torch.from_numpy((A[:, :, None] / (1j * w - E[:, :, None])).sum(1)).cuda()
    eps = torch.from_numpy(rng.uniform(-1, 1, n)).cuda()
    z = torch.zeros(n, dtype=torch.float64, device="cuda")
    ng = len(cpe_grid()) - 2
    seed = torch.rand(n, ng, dtype=torch.float32, device="cuda") + 0.5  # every weight in the support: 128 > 64 rows
    one = torch.ones(n, dtype=torch.float64, device="cuda")

    def run(lo, hi):
        e = torch.zeros(hi - lo, dtype=torch.float64, device="cuda")
        info = torch.full((hi - lo,), -9, dtype=torch.int32, device="cuda")
        if seeded:
            ctx.cpe_seed(seed[lo:hi].contiguous(), one[lo:hi].contiguous())
        ctx.continue_(gw.GW_CPE, S[lo:hi].contiguous(), eps[lo:hi].contiguous(), z[lo:hi].contiguous(),
                      z[lo:hi].contiguous(), None, None, e, info)
        ctx.sync()
        return e, info

    e, info = run(0, n)
    assert int(info.min()) >= 0  # no problem left to be done again
    for lo in range(0, n, 97):
        e1, i1 = run(lo, min(n, lo + 3))
        assert torch.equal(e1, e[lo:lo + 3]) and torch.equal(i1, info[lo:lo + 3])
    ctx.close()
