"""Loading the counts of few large patches uses the whole GPU, also where they are fractional (a calibrated
image) and each costs a float64 logarithm and lgamma: one source's five patches of 129 x 129 pixels take
less than a third of thirty such sources' time.  (One CTA per patch, 5 or 150 in all, made the two equal;
spread over the chip, the thirty have thirty times the work for the same 152 SMs.)"""
import copy
import dataclasses

import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu


def _sources(n):
    """n sources, each on five images of its own."""
    one = synth.single_source(seed=3, size=129)
    sc = copy.copy(one)
    sc.images = [dataclasses.replace(im, wcs=im.wcs + np.array([0, 0, 0, 0, -1000.0 * k, 0]))
                 for k in range(n) for im in one.images]
    sc.u0 = one.u0 + np.arange(n)[:, None] * np.array([[1000.0, 0.0]])
    sc.radius = np.repeat(one.radius, n).astype(np.int32)
    return sc


def test_fractional_counts_of_few_patches():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import paper_1611_03404_gb300 as P
    dev = torch.device("cuda:0")
    ms = {}
    for n in (1, 30):
        sc = _sources(n)
        px = [torch.as_tensor(im.pixels * np.float32(1.37), device=dev).contiguous() for im in sc.images]
        prob = P.Problem(sc, device=dev, device_pixels=px)
        assert prob.counts()["pixels"] == n * 5 * 129 * 129
        times = []
        for _ in range(20):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            torch.cuda.synchronize()
            a.record()
            prob.refresh_pixels()
            b.record()
            torch.cuda.synchronize()
            times.append(a.elapsed_time(b))
        ms[n] = float(np.median(times[5:]))
        prob.close()
    assert ms[1] < ms[30] / 3, ms
