"""The background's tile groups: few neighbours (staged once for several tiles) and more than one chunk of
them, in every tile size, rendered one tile per CTA and several, give the same bits and the oracle's ELBO."""
import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu

RADII = [22, 5, 17, 12, 20, 9, 22, 3, 18, 21, 14, 19]   # up to 2025 pixels; the first four alone: <= 8 neighbours
SHIFT = 4096.0


def _scene(n, copies):
    """n sources in one 64 x 64 image, `copies` of it side by side in the world.  Positions are multiples of
    2^-10 and the map is a shift, so that every copy's arithmetic is the same."""
    rng = np.random.default_rng(31)
    u = np.round(rng.uniform(22, 42, (n, 2)) * 1024) / 1024
    psf = synth._make_psf(rng, smooth=False)
    theta = np.stack([synth._initial_theta(rng, u[s], s % 2 == 0, [0.4, 0.6, 0.7, 1.5], 2.5, np.zeros(4), 0.0)
                      for s in range(n)])
    pixels = rng.poisson(90.0, (64, 64)).astype(np.float32)
    images, u0, th = [], [], []
    for c in range(copies):
        images.append(synth.Image(pixels, 2, 90.0, 200.0, np.array([1, 0, 0, 1, -SHIFT * c, 0.0]), psf))
        off = np.array([SHIFT * c, 0.0])
        u0.append(u + off)
        t = theta.copy()
        t[:, 0:2] = u + 0.25 + off
        th.append(t)
    return synth.Scene(images, np.concatenate(u0), np.array(RADII[:n] * copies, np.int32), np.concatenate(th),
                       synth.DEFAULT_PRIORS.copy())


@pytest.mark.parametrize("window", [False, True])
@pytest.mark.parametrize("n,tile", [(4, 128), (12, 128), (4, 256), (12, 256), (12, 512), (4, 1024)])
def test_grouped_tiles(n, tile, window):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import paper_1611_03404_gb300 as P
    dev = torch.device("cuda:0")
    n_sm = torch.cuda.get_device_properties(dev).multi_processor_count
    one = P.Problem(_scene(n, 1), device=dev, tile_pixels=tile).counts()["tiles"]
    many = 3 * n_sm * 32 // one + 1   # groups of three
    out = []
    for copies in (1, many):
        sc = _scene(n, copies)
        prob = P.Problem(sc, device=dev, tile_pixels=tile)
        assert (prob.counts()["tiles"] >= 3 * n_sm * 32) == (copies > 1)
        th = torch.as_tensor(sc.theta0, device=dev).contiguous()
        prob.render_background(th, **({"mode": P.NBR_WINDOW} if window else {}))
        out.append([t.reshape(copies, n, -1) for t in prob.elbo_batch(th)])
    for a, b in zip(*out):
        assert torch.isfinite(a).all()
        assert torch.equal(b, a.expand_as(b))
    if not window:
        from oracle.celeste_oracle import Oracle
        sc = _scene(n, 1)
        orc = Oracle(sc)
        for s in (0, n - 1):
            L = orc.elbo_grad_hess(s, sc.theta0[s], sc.theta0)[0]
            assert abs(float(out[0][0][0, s]) - L) <= 1e-6 * abs(L)
