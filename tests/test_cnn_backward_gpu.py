"""The backward GEMMs at batch sizes on both sides of their 64-row tiles and K splits: every layer's input and
weight gradient against float64 products of the BF16 operands the GPU used.  A stored input gradient
carries one BF16 rounding (half an ulp, 2^-9 of the entry) after a float32 sum of at most 576 products of
8-bit significands; a weight gradient is a float32 sum of up to 1024 B products, added in any order:
sqrt-law rounding n^(1/2) 2^-24 stays under 1e-5 of its norm up to B = 300."""
import numpy as np
import pytest
import torch
import torch.nn.functional as F

pytestmark = pytest.mark.gpu

SHAPES = [(32, 3, 3, 5), (64, 3, 3, 32), (64, 3, 3, 64), (64, 3, 3, 64), (256, 1024), (27, 256)]


def _f64(bits):
    return bits.view(torch.bfloat16).double()


@pytest.mark.parametrize("batch", [1, 3, 8, 17, 65, 300])
def test_gradients_of_every_layer(batch):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_1611_03404_gb300 import cnn
    dev = torch.device("cuda:0")
    net = cnn.WarmStartCNN(dev, seed=6)
    gen = torch.Generator(device=dev).manual_seed(batch)
    rand = lambda *s: torch.randn(*s, device=dev, dtype=torch.float32, generator=gen)
    net.params += 0.03 * rand(net.n)
    net.params_bf16.copy_(net.params.to(torch.bfloat16).view(torch.int16))
    x = rand(batch, 32, 32, 5).to(torch.bfloat16).view(torch.int16)
    dy = rand(batch, 27) / batch
    net.forward(x)
    net.grad.zero_()
    net.backward(x, dy)
    buf = {k: _f64(v) for k, v in net.buffers(batch).items()}
    w, b, at = [], [], 0
    for s in SHAPES:
        n = int(np.prod(s))
        w.append((at, n))
        b.append((at + n, s[0]))
        at += n + s[0]
    weight = lambda k: _f64(net.params_bf16[w[k][0]:w[k][0] + w[k][1]].contiguous()).view(SHAPES[k])
    act = [_f64(x)] + [buf[f"a{k}"] for k in range(1, 6)]
    d = [buf[f"d{k}"] for k in range(1, 6)] + [dy.to(torch.bfloat16).double()]   # d[k]: gradient at layer k's output
    for k in range(6):
        g = net.grad[w[k][0]:w[k][0] + w[k][1]].double().view(SHAPES[k])
        gb = net.grad[b[k][0]:b[k][0] + b[k][1]].double()
        if k < 4:
            a, o, wt = act[k].permute(0, 3, 1, 2), d[k].permute(0, 3, 1, 2), weight(k).permute(0, 3, 1, 2)
            st = 1 if k == 0 else 2
            ref = torch.nn.grad.conv2d_weight(a, wt.shape, o, stride=st, padding=1).permute(0, 2, 3, 1)
            if k:
                back = torch.nn.grad.conv2d_input(a.shape, wt, o, stride=st, padding=1)
                back = torch.where(a > 0, back, torch.zeros_like(back)).permute(0, 2, 3, 1)
        else:
            a = act[k].reshape(batch, -1)
            ref, back = d[k].T @ a, d[k] @ weight(k)
            back = torch.where(a > 0, back, torch.zeros_like(back)).view(act[k].shape)
        assert float((g - ref).norm()) <= 1e-5 * float(ref.norm()), k
        bias_ref = (dy.double() if k == 5 else d[k]).reshape(-1, SHAPES[k][0]).sum(0)
        scale = (dy.double() if k == 5 else d[k]).reshape(-1, SHAPES[k][0]).abs().sum(0)
        assert bool(((gb - bias_ref).abs() <= 1e-5 * scale + 1e-30).all()), k
        if k:
            got = d[k - 1]
            # half a BF16 ulp of the entry, plus float32 rounding of a sum that may cancel
            tol = 2.0 ** -8 * back.abs() + 1e-5 * back.abs().max()
            assert bool(((got - back).abs() <= tol).all()), k


def test_weights_off_a_16_byte_boundary():
    """The BF16 weights may start anywhere: same gradients as from an aligned copy."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_1611_03404_gb300 import cnn
    dev = torch.device("cuda:0")
    gen = torch.Generator(device=dev).manual_seed(2)
    x = torch.randn(5, 32, 32, 5, device=dev, dtype=torch.float32, generator=gen).to(torch.bfloat16).view(torch.int16)
    dy = torch.randn(5, 27, device=dev, dtype=torch.float32, generator=gen)
    net = cnn.WarmStartCNN(dev, seed=6)
    net.forward(x)
    net.grad.zero_()
    net.backward(x, dy)
    ref, d1 = net.grad.clone(), net.buffers(5)["d1"].clone()
    odd = torch.empty(net.n + 8, dtype=torch.int16, device=dev)[3:3 + net.n]
    odd.copy_(net.params_bf16)
    net.params_bf16 = odd
    net.grad.zero_()
    net.backward(x, dy)
    assert torch.equal(net.buffers(5)["d1"], d1)
    assert float((net.grad - ref).norm()) <= 1e-6 * float(ref.norm())   # (atomic additions in any order)
