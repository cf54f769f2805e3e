"""The backward pass with BF16 weights off a 16-byte boundary, at batch sizes whose last row tile is masked: the
16-byte copies then take their addresses from the workspace alone, and the input gradients are those
of an aligned copy bit for bit, the weight gradients up to the order of their atomic additions (float32 sums:
a few 2^-24 of a gradient's norm)."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batch", [1, 5, 65])
@pytest.mark.parametrize("shift", [1, 4, 7])
def test_backward_with_shifted_weights(batch, shift):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_1611_03404_gb300 import cnn
    dev = torch.device("cuda:0")
    gen = torch.Generator(device=dev).manual_seed(batch)
    x = torch.randn(batch, 32, 32, 5, device=dev, dtype=torch.float32, generator=gen).to(torch.bfloat16).view(torch.int16)
    dy = torch.randn(batch, 27, device=dev, dtype=torch.float32, generator=gen)
    net = cnn.WarmStartCNN(dev, seed=6)
    net.forward(x)
    net.grad.zero_()
    net.backward(x, dy)
    ref = net.grad.clone()
    d = {k: v.clone() for k, v in net.buffers(batch).items() if k[0] == "d"}
    aligned = net.params_bf16
    net.params_bf16 = torch.empty(net.n + 8, dtype=torch.int16, device=dev)[shift:shift + net.n]
    net.params_bf16.copy_(aligned)
    assert net.params_bf16.data_ptr() % 16 == 2 * shift
    net.grad.zero_()
    net.backward(x, dy)
    for k, v in d.items():
        assert torch.equal(net.buffers(batch)[k], v), k
    assert float((net.grad - ref).norm()) <= 1e-6 * float(ref.norm())
