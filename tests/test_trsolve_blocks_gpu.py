"""Trust-region subproblems whose reduction has nothing to reflect in some columns (diagonal matrices,
blocks, a single coupled pair): both solver layouts against the oracle."""
import numpy as np
import pytest
import torch

from test_trsolve_gpu import _check_against_oracle

pytestmark = pytest.mark.gpu


def _matrix(kind, rng):
    B = np.diag(rng.uniform(0.5, 3.0, 27) * rng.choice([-0.2, 1.0], 27, p=[0.2, 0.8]))
    if kind == "first":      # a dense leading block, nothing below it
        M = rng.normal(size=(9, 9))
        B[:9, :9] += 0.3 * (M + M.T)
    elif kind == "last":     # only the last columns couple
        M = rng.normal(size=(4, 4))
        B[23:, 23:] += 0.3 * (M + M.T)
    elif kind == "pair":
        B[25, 26] = B[26, 25] = 0.7
        B[3, 20] = B[20, 3] = -0.4
    elif kind == "tiny":     # couplings whose squares underflow
        B[np.arange(26), np.arange(1, 27)] = B[np.arange(1, 27), np.arange(26)] = 1e-170
    return B


@pytest.mark.parametrize("warps", [1, 4])
@pytest.mark.parametrize("kind", ["diagonal", "first", "last", "pair", "tiny"])
def test_subproblem_without_couplings(kind, warps):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import paper_1611_03404_gb300 as P
    rng = np.random.default_rng(31)
    B = np.array([_matrix(kind, rng) for _ in range(24)])
    g = rng.normal(size=(24, 27)) * rng.choice([1e-2, 1.0, 30.0], (24, 1))
    d = rng.choice([0.05, 1.0, 20.0, 1e4], 24)
    dev = [torch.as_tensor(a, device="cuda:0").contiguous() for a in (B, g, d)]
    p, pred, _ = P.tr_solve_batch(*dev, warps=warps)
    _check_against_oracle(B, g, d, p.cpu().numpy(), pred.cpu().numpy())
