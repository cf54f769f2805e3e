"""The network's bounded waits run out: with budgets from none at all to a few microseconds, whichever of the
tcgen05 kernels' roles gives up first (producers, products, epilogue; between a CTA's first tile and its last
image), the call ends, celeste_cnn_status reports it, and the next call with the default budget gives the
same bits as before.  900 patches are three images of the first layer for every CTA of an SM's two."""
import ctypes

import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batch", [1, 900])
@pytest.mark.parametrize("budget", [-1, 1, 300, 1000, 2000, 4000, 8000, 16000, 40000])
def test_waits_that_run_out(batch, budget):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import paper_1611_03404_gb300 as P
    from paper_1611_03404_gb300 import cnn
    dev = torch.device("cuda:0")
    net = cnn.WarmStartCNN(dev, seed=6)
    gen = torch.Generator(device=dev).manual_seed(batch)
    x = torch.randn(batch, 32, 32, 5, device=dev, dtype=torch.float32, generator=gen).to(torch.bfloat16).view(torch.int16)
    ref = net.forward(x)
    assert P.lib().celeste_cnn_status() == 0
    _, ws, nb = net.workspace(batch)
    y = torch.empty_like(ref)
    ptr = lambda t: ctypes.c_void_p(t.data_ptr())
    for _ in range(4):
        rc = P.lib().celeste_cnn_forward_budget(
            ptr(net.params), ptr(net.params_bf16), ptr(x), batch, None, None, ptr(y), ws, ctypes.c_size_t(nb),
            cnn.ENGINE_TCGEN05, budget, ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
        assert rc == 0
        status = P.lib().celeste_cnn_status()
        assert status in (0, 3)                      # ok, or a wait that ran out
        if budget < 0:
            assert status == 3
        if status == 0:
            assert torch.equal(y, ref)
        assert P.lib().celeste_cnn_status() == 0     # (reported once)
    assert torch.equal(net.forward(x), ref)
    assert P.lib().celeste_cnn_status() == 0
