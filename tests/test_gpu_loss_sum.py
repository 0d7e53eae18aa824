"""The training loss is summed beyond FP32: over many equal samples it is that of one."""
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n", [40000, 1 << 22])
def test_equal_samples(n):
    from paper_2002_04353_gb300 import alelb
    net = alelb.Mlp(seed=5)
    d = torch.device("cuda")
    one = (torch.tensor([[0.3, -0.7, 0.1, 0.9, -0.2, 0.5]], device=d), torch.tensor([4], dtype=torch.int16, device=d),
           torch.tensor([[0.2, 0.5, 0.3]], device=d), torch.tensor([9], dtype=torch.uint8, device=d))
    single, _ = net.loss_grad(*one, w_bary=0.5)
    many, _ = net.loss_grad(*(v.expand(n, *v.shape[1:]).contiguous() for v in one), w_bary=0.5)
    # the sample's own terms, and the sum of a few samples, in FP32: some eight roundings of 2^-24
    assert abs(many - single) <= 8 * 2.0 ** -24 * abs(single)
