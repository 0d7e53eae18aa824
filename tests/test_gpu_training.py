"""Loss and gradient of the element proposal at the sizes where the tiling can go wrong (one sample, around a tile of 32, more tiles
than blocks), against the same network in FP64, and training that repeats bit for bit."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _data(n, seed=0):
    gen = torch.Generator().manual_seed(seed)
    feat = torch.rand((n, 6), generator=gen) * 2 - 1
    ring = torch.randint(1, 33, (n,), generator=gen)
    slot = (torch.rand(n, generator=gen) * ring).long().clamp(max=31)
    slot = torch.minimum(slot, ring - 1)
    bary = torch.rand((n, 3), generator=gen)
    d = torch.device("cuda")
    return feat.to(d), slot.to(torch.int16).to(d), bary.to(d), ring.to(torch.uint8).to(d)


def _reference(h, feat, slot, bary, ring, w):
    at = np.cumsum([0, 384, 64, 4096, 64, 2240, 35])
    h = torch.from_numpy(h).double().cuda().requires_grad_(True)
    W1, b1, W2, b2, W3, b3 = (h[at[j]:at[j + 1]] for j in range(6))
    z = torch.tanh(feat.double() @ W1.view(64, 6).T + b1)
    z = torch.tanh(z @ W2.view(64, 64).T + b2)
    o = z @ W3.view(35, 64).T + b3
    dead = torch.arange(32, device="cuda")[None] >= ring.long()[:, None]
    ce = torch.nn.functional.cross_entropy(o[:, :32].masked_fill(dead, -float("inf")), slot.long(), reduction="none")
    loss = (ce + w * ((o[:, 32:] - bary.double()) ** 2).mean(1)).mean()
    g, = torch.autograd.grad(loss, h)
    return float(loss), g.cpu().numpy()


@pytest.mark.parametrize("n", [1, 31, 32, 33, 1000, 9728, 9729, 40000])
def test_loss_and_gradient(n):
    from paper_2002_04353_gb300 import alelb
    net = alelb.Mlp(seed=5)
    d = _data(n, seed=n)
    loss, g = net.loss_grad(*d, w_bary=0.5)
    lr, gr = _reference(net.params(rounded=True), *d, 0.5)
    # FP32 sums of at most 40000 terms in 32 x 64 x 304 partial sums: a few 1e-6 of the gradient's norm
    assert abs(loss - lr) <= 2e-6 * abs(lr)
    assert np.linalg.norm(g - gr) <= 1e-5 * np.linalg.norm(gr)


def test_training_repeats_bit_for_bit():
    from paper_2002_04353_gb300 import alelb
    d = _data(20001, seed=9)
    out = []
    for _ in range(2):
        net = alelb.Mlp(seed=3)
        loss = net.train(*d, epochs=2, batch=1111, lr=2e-3, w_bary=0.5, seed=7)
        out.append((loss, net.params()))
    assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1])
