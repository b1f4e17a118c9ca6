"""Loss and gradients of the seed network at the edges of its GEMM tiles: one 128-sample block, parts of the
batch that end early, more than 16 parts' worth of samples, hidden layers of one and three 128-row tiles,
an input of one 64-wide tile; against 64-bit sums over the operands as the kernels round them (weights,
activations and dZ in fp16). What remains is FP32 accumulation, up to 256 2^-24 of a sum, which turns up to
3 % of the fp16 roundings the other way: sqrt(0.03) 2^-11 per operand, eight operands in quadrature."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batch,nin,nh,nhidden", [(128, 64, 128, 1), (384, 128, 384, 2), (4736, 128, 256, 3), (640, 192, 128, 4)])
def test_loss_grad(batch, nin, nh, nhidden):
    import torch

    import paper_1602_02313_gb300 as gw
    from paper_1602_02313_gb300 import build as b
    b.build()
    rng = np.random.default_rng(batch)
    f16 = lambda a: np.asarray(a, np.float32).astype(np.float16).astype(np.float32)  # noqa: E731
    net = gw.MLP(nin=nin, nh=nh, nhidden=nhidden, nout=128, seed=5)
    net.set_params(f16(net.get_params() + 0.01 * rng.standard_normal(net.num_params()).astype(np.float32)))
    x, A = f16(0.5 * rng.standard_normal((batch, nin))), f16(0.05 * rng.standard_normal((nin, 128)))
    loss = torch.zeros(1, dtype=torch.float32, device="cuda")
    grads = torch.zeros(net.num_params(), dtype=torch.float32, device="cuda")
    for _ in range(2):  # the second call finds the workspaces of the first
        net.loss_grad(torch.from_numpy(x).cuda(), torch.from_numpy(A).cuda(), loss, grads)
    net.sync()
    d = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda().double()  # noqa: E731
    half = lambda t: t.half().double()  # noqa: E731
    p, sizes, off, W, B = net.get_params(), [nin] + [nh] * nhidden + [128], 0, [], []
    for di, do in zip(sizes[:-1], sizes[1:]):
        W.append(half(d(p[off:off + di * do].reshape(do, di))))
        B.append(d(p[off + di * do:off + di * do + do]))
        off += di * do + do
    hs, zs, xd, Ad = [half(d(x))], [], d(x), d(A)
    for i in range(nhidden + 1):
        z = hs[-1] @ W[i].T + B[i]
        zs.append(z)
        hs.append(half(torch.nn.functional.gelu(z)) if i < nhidden else torch.nn.functional.softplus(z, threshold=1e9))
    r = hs[-1] @ Ad.T - xd
    assert abs(float(loss) - float(r.square().sum()) / batch) < 1e-4 * float(r.square().sum()) / batch
    dz = (2.0 / batch) * (r @ Ad) * torch.sigmoid(zs[-1])
    off = net.num_params()
    for i in range(nhidden, -1, -1):
        want = torch.cat([(half(dz).T @ hs[i]).reshape(-1), dz.sum(0)])
        off -= want.numel()
        got = grads[off:off + want.numel()].double()
        assert float((got - want).norm()) < np.sqrt(8 * 0.03) * 2.0 ** -11 * float(want.norm())
        if i:
            z = zs[i - 1]
            dgelu = 0.5 * (1 + torch.erf(z / 2 ** 0.5)) + z * torch.exp(-0.5 * z * z) / (2 * np.pi) ** 0.5
            dz = (half(dz) @ W[i]) * dgelu
    net.close()
