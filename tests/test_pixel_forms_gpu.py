"""The pixel kernel's forms at patch sizes on both sides of its 32-pixel slices and of its tiles: patches
evaluated one tile per CTA and as the second or later tile of a persistent CTA give the same bits, and
the ELBO matches the oracle."""
import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu

RADII = [1, 2, 3, 4, 5, 8, 11, 12, 17, 22]   # 9 .. 2025 pixels: ragged slices, full slices, several tiles
COPIES = 80
SHIFT = 4096.0


def _scene(copies):
    """RADII's sources in one 64 x 64 image, and `copies` of it side by side in the world.  Positions are
    multiples of 2^-10 and the map is a shift, so that every copy's arithmetic is the same."""
    rng = np.random.default_rng(77)
    S = len(RADII)
    u = np.round(rng.uniform(14, 50, (S, 2)) * 1024) / 1024
    psf = synth._make_psf(rng, smooth=False)
    theta = np.stack([synth._initial_theta(rng, u[s], s % 2 == 0, [0.4, 0.6, 0.7, 1.5], 2.5, np.zeros(4), 0.0)
                      for s in range(S)])
    pixels = rng.poisson(90.0, (64, 64)).astype(np.float32)
    images, u0, th = [], [], []
    for c in range(copies):
        images.append(synth.Image(pixels, 2, 90.0, 200.0, np.array([1, 0, 0, 1, -SHIFT * c, 0.0]), psf))
        off = np.array([SHIFT * c, 0.0])
        u0.append(u + off)
        t = theta.copy()
        t[:, 0:2] = u + 0.25 + off
        th.append(t)
    return synth.Scene(images, np.concatenate(u0), np.array(RADII * copies, np.int32), np.concatenate(th),
                       synth.DEFAULT_PRIORS.copy())


@pytest.mark.parametrize("tile,hessian", [(128, 0), (128, 1), (128, 2), (128, 3), (128, 4), (256, 0), (512, 0), (1024, 0)])
def test_first_and_later_tiles_give_the_same_bits(tile, hessian):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import paper_1611_03404_gb300 as P
    dev = torch.device("cuda:0")
    out = []
    for copies in (1, COPIES):
        sc = _scene(copies)
        prob = P.Problem(sc, device=dev, tile_pixels=tile, hessian_mode=hessian)
        n_sm = torch.cuda.get_device_properties(dev).multi_processor_count
        assert (prob.counts()["tiles"] > 5 * n_sm) == (copies > 1)
        th = torch.as_tensor(sc.theta0, device=dev).contiguous()
        prob.render_background(th)
        out.append([t.reshape(copies, len(RADII), -1) for t in prob.elbo_batch(th)])
    for one, many in zip(*out):
        assert torch.isfinite(one).all()
        for c in (0, 1, COPIES // 2, COPIES - 1):
            assert torch.equal(many[c], one[0])
    from oracle.celeste_oracle import Oracle
    sc = _scene(1)
    orc = Oracle(sc)
    for s in (0, 4, len(RADII) - 1):
        L = orc.elbo_grad_hess(s, sc.theta0[s], sc.theta0)[0]
        assert abs(float(out[0][0][0, s]) - L) <= 1e-6 * abs(L)
