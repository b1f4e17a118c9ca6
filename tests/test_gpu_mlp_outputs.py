"""Loss and gradients of the seed network with more outputs than shared memory holds (very fine pole grids): the loss
kernel then takes one sample per block and reads its outputs from memory. Against 64-bit sums over the operands as the
kernels round them, with the tolerance of test_gpu_mlp_tiles.py (eight fp16 operands of which 3 % round the other way)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nout", [6400, 58240])
def test_many_outputs(nout):
    import torch

    import paper_1602_02313_gb300 as gw
    from paper_1602_02313_gb300 import build as b
    b.build()
    B, nin, nh = 128, 64, 128
    rng = np.random.default_rng(nout)
    f16 = lambda a: np.asarray(a, np.float32).astype(np.float16).astype(np.float32)  # noqa: E731
    net = gw.MLP(nin=nin, nh=nh, nhidden=1, nout=nout, seed=5)
    p = f16(net.get_params())
    net.set_params(p)
    x, A = f16(0.5 * rng.standard_normal((B, nin))), f16(rng.standard_normal((nin, nout)) / np.sqrt(nout))
    loss = torch.zeros(1, dtype=torch.float32, device="cuda")
    grads = torch.zeros(net.num_params(), dtype=torch.float32, device="cuda")
    net.loss_grad(torch.from_numpy(x).cuda(), torch.from_numpy(A).cuda(), loss, grads)
    net.sync()
    d = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda().double()  # noqa: E731
    half = lambda t: t.half().double()  # noqa: E731
    n0 = nin * nh
    W0, b0 = d(p[:n0].reshape(nh, nin)), d(p[n0:n0 + nh])
    n1 = n0 + nh
    W1, b1 = d(p[n1:n1 + nh * nout].reshape(nout, nh)), d(p[n1 + nh * nout:])
    xd, Ad = d(x), d(A)
    z0 = xd @ W0.T + b0
    h0 = half(torch.nn.functional.gelu(z0))
    z1 = h0 @ W1.T + b1
    r = torch.nn.functional.softplus(z1, threshold=1e9) @ Ad.T - xd
    want = float(r.square().sum()) / B
    assert abs(float(loss) - want) < 1e-4 * want
    dz1 = (2.0 / B) * (r @ Ad) * torch.sigmoid(z1)
    dgelu = 0.5 * (1 + torch.erf(z0 / 2 ** 0.5)) + z0 * torch.exp(-0.5 * z0 * z0) / (2 * np.pi) ** 0.5
    dz0 = (half(dz1) @ W1) * dgelu
    tol = np.sqrt(8 * 0.03) * 2.0 ** -11
    for got, dz, h in ((grads[:n1], dz0, xd), (grads[n1:], dz1, h0)):
        ref = torch.cat([(half(dz).T @ h).reshape(-1), dz.sum(0)])
        assert float((got.double() - ref).norm()) < tol * float(ref.norm())
    net.close()
