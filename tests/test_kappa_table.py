"""The log-factorial terms' table of a problem: no larger than its pixels need, and the same bits as the terms
evaluated per pixel on both sides of its edge.

A source's ELBO does not depend on what else is in its problem, but the table does: with a second source far
away the problem has more pixels and the table more entries.  The counts lie within +-8 of an edge that the
smaller problem's table ends at or before, so the two runs take a pixel's term from the table and from its
evaluation; every float32 sum has the same operands in the same order, and the results have to be equal.  Wrong entries
show: the sky lies at the edge and the sources are faint, so that a tile's sum is a few hundred at a float32
spacing of 3e-5 to 6e-5, and an index off by one count shifts it by 128 / (2 edge), 1e-3 or more."""
import copy

import numpy as np
import pytest
import torch

import synth


def _scene(radius, edge, others):
    """One source of five patches; `others` more, each 1000 pixels further along in a larger image."""
    one = synth.single_source(seed=8, size=2 * radius + 1)
    size = one.images[0].H
    sc = copy.copy(one)
    rng = np.random.default_rng(3)
    for im in sc.images:
        im.sky, im.iota = float(edge), 1.0
        px = rng.integers(edge - 8, edge + 9, (size, size))
        im.pixels = np.full((size, size + 1000 * others), edge, np.float32)
        im.pixels[:, :size] = px
    shift = np.arange(others + 1)[:, None] * 1000.0
    sc.u0 = np.repeat(one.u0, others + 1, 0)
    sc.u0[:, :1] += shift
    sc.theta0 = np.repeat(one.theta0, others + 1, 0)
    sc.theta0[:, 7] = sc.theta0[:, 9] = -6.0      # mean flux e^-6
    sc.theta0[:, :1] += shift
    sc.radius = np.repeat(one.radius, others + 1).astype(np.int32)
    return sc


def test_workspace_of_a_small_problem():
    """49 pixels: everything else in the workspace is under 100 KB, a full table alone would be 256 KB."""
    import __graft_entry__
    __graft_entry__.build()
    import paper_1611_03404_gb300 as P
    sc = synth.tiny(seed=1, n_sources=1, n_images=1, radius=(3, 3))
    assert P.HostProblem(sc).workspace_bytes() < 4 * 65536


# (radius, edge, other sources): alone, a source's table has as many entries as its pixels; one more source
# doubles them, eight more fill the table
@pytest.mark.gpu
@pytest.mark.parametrize("radius,edge,others", [(1, 45, 1), (20, 8405, 1), (20, 65536, 8)])
def test_same_bits_around_the_edge(radius, edge, others):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import paper_1611_03404_gb300 as P
    dev = torch.device("cuda:0")
    elbo, entries = [], []
    for k in (0, others):
        sc = _scene(radius, edge, k)
        th = torch.as_tensor(sc.theta0, device=dev).contiguous()
        prob = P.Problem(sc, device=dev)
        entries.append(min(prob.counts()["pixels"], 65536))
        prob.render_background(th)
        elbo.append([float(prob.elbo_batch(th, want=w)[0][0]) for w in (P.WANT_ELBO, P.WANT_ELBO | P.WANT_GRAD)])
    assert entries[0] < edge + 8 and entries[1] >= min(edge + 9, 65536)
    assert elbo[0] == elbo[1]
