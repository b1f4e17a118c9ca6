"""Loss and gradients of the seed network where memory is short: one layer's dZ at a time and no parts of the weight
gradients. The chain of dZ, and with it the bias gradients, keeps its bits; the weight gradients are one FP32 chain of
128 MMAs over the batch instead of eight of 16, summed: each within 128 2^-23 of the sum of the terms' magnitudes, about
sqrt(2048) times the sum itself. The rest of the memory is held by a tensor that nothing touches."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

MIB = 1 << 20


def test_short_of_memory():
    import torch

    import paper_1602_02313_gb300 as gw
    from paper_1602_02313_gb300 import build as b
    b.build()
    batch, nin, nh, nhidden, nout = 2048, 128, 2048, 4, 128
    # 13.1 M parameters: eight parts 420 MiB, activations 134, dZ of every layer 135, dZ of one layer 40
    rng = np.random.default_rng(3)
    x = torch.from_numpy(rng.standard_normal((batch, nin)).astype(np.float32)).cuda()
    A = torch.from_numpy((0.1 * rng.standard_normal((nin, nout))).astype(np.float32)).cuda()
    loss = [torch.zeros(1, dtype=torch.float32, device="cuda") for _ in range(2)]
    nets = [gw.MLP(nin=nin, nh=nh, nhidden=nhidden, nout=nout, seed=9) for _ in range(2)]
    grads = [torch.zeros(nets[0].num_params(), dtype=torch.float32, device="cuda") for _ in range(2)]
    nets[0].loss_grad(x, A, loss[0], grads[0])
    nets[0].sync()
    torch.cuda.synchronize()
    hold = []  # down to 330 MiB, in pieces as large as can be had
    while (n := torch.cuda.mem_get_info()[0] // MIB - 330) > 0:
        for part in (n, n // 2, n // 8, 2):
            try:
                hold.append(torch.empty(part * MIB, dtype=torch.uint8, device="cuda"))
                break
            except torch.OutOfMemoryError:
                assert part > 2
        else:
            break
    try:
        nets[1].loss_grad(x, A, loss[1], grads[1])
        nets[1].loss_grad(x[:1024], A, loss[1], grads[1])  # a smaller batch in the same workspace
        nets[1].loss_grad(x, A, loss[1], grads[1])
        nets[1].sync()
    finally:
        del hold
        torch.cuda.empty_cache()
    assert abs(float(loss[1] - loss[0])) < 1e-5 * float(loss[0])  # summed by atomics
    sizes, off = [nin] + [nh] * nhidden + [nout], 0
    for di, do in zip(sizes[:-1], sizes[1:]):
        w, bias = slice(off, off + di * do), slice(off + di * do, off + di * do + do)
        off += di * do + do
        assert torch.equal(grads[0][bias], grads[1][bias])
        ref = grads[0][w].double()
        assert float((grads[1][w].double() - ref).norm()) < 2 * 128 * 2.0 ** -23 * 2048 ** 0.5 * float(ref.norm())
    for net in nets:
        net.close()
