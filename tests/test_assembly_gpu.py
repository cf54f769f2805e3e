"""Assembly of a source's ELBO, gradient and Hessian from one to many patches (fewer and more than the
kernel's warps take at a time), with one and with several tiles per patch, against the oracle."""
import numpy as np
import pytest
import torch

import synth
from oracle import celeste_oracle as O
from test_parity_gpu import check_elbo, check_grad, check_hess, grad_natural_scale, hess_natural_scale

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_images", [1, 2, 4, 5, 8, 9, 13, 17])
def test_patch_counts(n_images):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import paper_1611_03404_gb300 as P
    sc = synth.tiny(seed=40 + n_images, n_sources=2, n_images=n_images, radius=(4, 9))
    dev = torch.device("cuda:0")
    prob = P.Problem(sc, device=dev)
    assert prob.counts()["patches"] == 2 * n_images
    th = torch.as_tensor(sc.theta0, device=dev).contiguous()
    prob.render_background(th)
    elbo, grad, hess = (t.cpu().numpy() for t in prob.elbo_batch(th))
    orc = O.Oracle(sc)
    for s in range(2):
        L, g, H = orc.elbo_grad_hess(s, sc.theta0[s], sc.theta0)
        check_elbo(elbo[s], L, f"{n_images} images, source {s}")
        check_grad(grad[s], g, f"{n_images} images, source {s}",
                   natural=lambda: grad_natural_scale(orc, s, sc.theta0[s], sc.theta0))
        check_hess(hess[s], H, f"{n_images} images, source {s}",
                   natural=lambda: hess_natural_scale(orc, s, sc.theta0[s], sc.theta0))
        assert np.array_equal(hess[s][2:, 2:], hess[s][2:, 2:].T)
