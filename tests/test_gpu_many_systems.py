"""The BF16 path with more systems than 65,535 groups of eight: the vector update's groups must not
be counted in a grid dimension of 16 bits.
"""
import numpy as np
import pytest
import torch

from oracle import filter as F
from paper_2503_00253_gb300 import workloads
from parity_checks import increment_error, mean_error

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ritz_rank", [10, 20])
def test_half_a_million_systems(ritz_rank):
    """128 members at 4097 nodes (524,417 systems) on a small grid; bound of the BF16 parity tests. Above rank
    15 a group is eight systems."""
    from paper_2503_00253_gb300 import binding as B
    grid = workloads.Grid((16, 16, 1), (True, True, False), (3.0, 3.0, 1.0), True)
    pr = workloads.random_obs_problem(grid, N=128, d=40, r2=0.8, Q=4097, tol=1e-6, seed=8)
    args = [torch.tensor(a, device="cuda") for a in (pr.X, pr.obs_idx, pr.y, pr.R)]
    mu, A, st = B.info_esrf_analysis(pr.grid, *args, pr.Q, pr.tol, B.make_options(precision=2, ritz_rank=ritz_rank))
    assert st["status"] == 0 and st["n_systems"] == 128 * 4097 + 1
    A_ref = F.perturbation_update(pr.X, pr.obs_idx, pr.R, pr.grid, pr.Q)
    assert increment_error(A, A_ref, pr.X - pr.X.mean(0)) <= 1e-4
    assert mean_error(mu, F.mean_update(pr.X, pr.obs_idx, pr.y, pr.R, pr.grid), pr.X.mean(0)) <= 1e-4
