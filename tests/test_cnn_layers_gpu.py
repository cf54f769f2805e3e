"""The tensor-core forward at batch sizes on both sides of its 128-row tiles and of the CTAs' shares, and
from an input that does not start on a 16-byte boundary: every layer's activations are the mma.sync
engine's (both add the same products in the same order)."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batch", [1, 2, 3, 7, 9, 33, 127, 129, 305, 700])
@pytest.mark.parametrize("offset", [0, 3])
def test_layers_match_the_other_engine(batch, offset):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_1611_03404_gb300 import cnn
    from paper_1611_03404_gb300.celeste import lib
    dev = torch.device("cuda:0")
    net = cnn.WarmStartCNN(dev, seed=3)
    gen = torch.Generator(device=dev).manual_seed(batch)
    net.params += 0.05 * torch.randn(net.n, device=dev, dtype=torch.float32, generator=gen)
    net.params_bf16.copy_(net.params.to(torch.bfloat16).view(torch.int16))
    net.set_standardisation(torch.randn(64, 27, device=dev, dtype=torch.float32, generator=gen))
    flat = torch.randn(batch * 5120 + 8, device=dev, dtype=torch.float32, generator=gen)
    flat = flat.to(torch.bfloat16).view(torch.int16)
    x = flat[offset:offset + batch * 5120].view(batch, 32, 32, 5)
    kept = {}
    for engine in (cnn.ENGINE_MMA_SYNC, cnn.ENGINE_TCGEN05):
        y = [net.forward(x, standardised=s, engine=engine).clone() for s in (True, False)]
        kept[engine] = y + [v.clone() for k, v in sorted(net.buffers(batch).items()) if k[0] == "a"]
    assert lib().celeste_cnn_status() == 0
    for a, b in zip(kept[cnn.ENGINE_MMA_SYNC], kept[cnn.ENGINE_TCGEN05]):
        assert torch.equal(a, b)
