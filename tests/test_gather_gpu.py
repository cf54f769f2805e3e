"""Log-factorial terms of the gathered counts: whole counts inside and beyond the table, calibrated
(fractional) counts and zeros give the same ELBO as the oracle; a bad count is still reported; new counts in
the same images replace the old ones."""
import numpy as np
import pytest
import torch

import synth
from oracle.celeste_oracle import Oracle

pytestmark = pytest.mark.gpu


def _scene(kind):
    sc = synth.tiny(seed=12, n_sources=2, n_images=2, rotate=False)
    rng = np.random.default_rng(5)
    for im in sc.images:
        if kind == "fractional":
            im.pixels = (im.pixels * 1.37).astype(np.float32)
        elif kind == "large":
            im.pixels = rng.integers(65530, 65545, im.pixels.shape).astype(np.float32)
        elif kind == "zeros":
            im.pixels = np.where(rng.random(im.pixels.shape) < 0.5, 0.0, im.pixels).astype(np.float32)
    return sc


@pytest.mark.parametrize("kind", ["whole", "fractional", "large", "zeros"])
def test_counts(kind):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import paper_1611_03404_gb300 as P
    dev = torch.device("cuda:0")
    sc, first = _scene(kind), _scene("whole")
    pixels = [torch.as_tensor(im.pixels, device=dev).contiguous() for im in first.images]
    prob = P.Problem(first, device=dev, device_pixels=pixels)
    for p, im in zip(prob.pixels, sc.images):
        p.copy_(torch.as_tensor(im.pixels, device=dev))
    prob.refresh_pixels()
    th = torch.as_tensor(sc.theta0, device=dev).contiguous()
    prob.render_background(th)
    elbo, _, _ = prob.elbo_batch(th)
    orc = Oracle(sc)
    for s in range(sc.n_sources):
        L = orc.elbo_grad_hess(s, sc.theta0[s], sc.theta0)[0]
        assert abs(float(elbo[s]) - L) <= 1e-6 * abs(L)
    prob.pixels[0].fill_(-1.0)
    prob.refresh_pixels()
    with pytest.raises(P.CelesteError):
        prob.check()
