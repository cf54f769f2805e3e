"""Light of a galaxy component under 2^-126 of its peak: it counts where the brightness constants, which
float32 holds up to 3.4e38, bring it back to counts.  A galaxy of mean flux e^88 lies a little over 13.2 PSF
widths from the pixel column nearest to it (exponent -126.5 in base 2; -142 and beyond in the other columns), so
that the column's rate is a few hundred counts over the sky; once as the evaluated source and once as a
neighbour's background, against the float64 oracle.

Tolerance: the light may be off by 1e-3 of itself: float32 keeps each of the 42 components' values near
1e-39 to 2^-150 (6e-5 of their sum) and their exponents of 127 to 2^-18 (4e-6); the means' and precisions' float32
rounding moves the exponent by 127 * 3 * 2^-23 (5e-5).  On the ELBO that is the change that a shift of the mean
log flux by 1e-3 makes, plus the usual 1e-6."""
import numpy as np
import pytest
import torch

import synth
from oracle.celeste_oracle import Oracle

pytestmark = pytest.mark.gpu
LOG_FLUX = 88.0


def _scene():
    sc = synth.tiny(seed=4, n_sources=2, n_images=1, H=40, W=40, radius=(1, 1), rotate=False)
    im = sc.images[0]
    im.wcs = np.array([1.0, 0, 0, 1.0, 0, 0])
    im.band = 2
    im.sky, im.iota = 90.0, 1000.0
    im.psf = np.zeros_like(im.psf)           # three equal round components of width 1 at the centre
    sc.u0 = np.array([[10.0, 20.0], [11.0, 20.0]])
    th = sc.theta0.copy()
    th[:, 0:2] = sc.u0
    th[:, 2] = -20.0                         # exponential profile
    th[:, 3:5] = 2.0, 0.3
    th[:, 5] = -6.0                          # a point: every component as wide as the PSF
    im.pixels = np.full((40, 40), 300.0, np.float32)
    return sc, th


def _bright(th, s, column):
    """Source s as the bright galaxy, its centre to the right of pixel column `column`."""
    th[s, 0] = column + np.sqrt(2.0 * np.log(2.0) * 126.5)
    th[s, 1] = 20.0
    th[s, 6] = 40.0
    th[s, 9], th[s, 10] = LOG_FLUX, -35.0
    th[s, 19:23], th[s, 23:27] = 0.0, -35.0
    return th


@pytest.mark.parametrize("role", ["source", "neighbour"])
@pytest.mark.parametrize("tile", [128, 256])
def test_light_below_the_normal_range(role, tile):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import paper_1611_03404_gb300 as P
    dev = torch.device("cuda:0")
    sc, th = _scene()
    bright = 0 if role == "source" else 1
    th = _bright(th, bright, 11)             # source 0's patch: columns 9 to 11
    orc = Oracle(sc)
    ref = orc.elbo_grad_hess(0, th[0], th)[0]
    off = th.copy()
    off[bright, 9] += 1e-3
    tol = abs(orc.elbo_grad_hess(0, off[0], off)[0] - ref) + 1e-6 * abs(ref)
    dark = th.copy()
    dark[bright, 9] -= 20.0                  # the same without that light (and its own KL term)
    if role == "neighbour":
        assert abs(orc.elbo_grad_hess(0, dark[0], dark)[0] - ref) > 100 * tol
    prob = P.Problem(sc, device=dev, tile_pixels=tile)
    t = torch.as_tensor(th, device=dev).contiguous()
    prob.render_background(t)
    full = prob.elbo_batch(t)[0]
    value = prob.elbo_batch(t, want=P.WANT_ELBO)[0]
    assert abs(float(full[0]) - ref) <= tol
    assert abs(float(value[0]) - ref) <= tol
