"""Sizes at which the general PCG kernel, the eigensolver, the weighted-sum operators and the
BF16 loop change their way of working, against the FP64 oracle.

Bounds: those of the end-to-end parity tests (FP64 1e-10 at PCG tolerance 1e-12, FP32 and
BF16 1e-4 at 1e-6).
"""
import dataclasses

import numpy as np
import pytest
import torch

from oracle import filter as F
from paper_2503_00253_gb300 import workloads
from parity_checks import increment_error, mean_error

pytestmark = pytest.mark.gpu

BOUND = {0: (1e-12, 1e-10), 1: (1e-6, 1e-4), 2: (1e-6, 1e-4)}


@pytest.fixture(scope="module")
def B():
    from paper_2503_00253_gb300 import binding
    binding.library()
    return binding


def dev(a):
    return torch.tensor(np.ascontiguousarray(a), device="cuda")


def check(B, pr, precision, **kw):
    """Analysis of pr within the precision's bound."""
    tol, bound = BOUND[precision]
    mu_a, A_a, st = B.info_esrf_analysis(pr.grid, dev(pr.X), dev(pr.obs_idx), dev(pr.y), dev(pr.R), pr.Q, tol,
                                         B.make_options(precision=precision, **kw))
    torch.cuda.synchronize()
    assert st["status"] == 0 and st["n_unconverged"] == 0, st
    A_ref = F.perturbation_update(pr.X, pr.obs_idx, pr.R, pr.grid, pr.Q)
    mu_ref = F.mean_update(pr.X, pr.obs_idx, pr.y, pr.R, pr.grid)
    assert increment_error(A_a, A_ref, pr.X - pr.X.mean(0)) <= bound
    assert mean_error(mu_a, mu_ref, pr.X.mean(0)) <= bound


def layered(d, N, nx, nz, c, Q, seed):
    grid = workloads.Grid((nx, 1, nz), (True, False, False), (c, 1.0, 1.5), True)
    return workloads.random_obs_problem(grid, N=N, d=d, r2=0.8, Q=Q, tol=1e-6, seed=seed)


# groups of two (FP64) and eight (FP32) systems; blocks of eight rows; 1024 rows staged at a time; FP32 vectors
# in shared memory up to 1551 rows, the direction alone up to 4778; FP64 up to 3200
@pytest.mark.parametrize("d,N,precision", [
    (1, 3, 1), (7, 9, 1), (8, 8, 1), (9, 2, 1), (63, 17, 1), (513, 8, 1), (1551, 3, 1), (1552, 3, 1), (2049, 7, 1),
    (4779, 3, 1), (1, 3, 0), (2, 2, 0), (33, 5, 0), (1025, 3, 0), (3200, 3, 0), (3201, 3, 0)])
def test_general_pcg_sizes(B, d, N, precision):
    check(B, layered(d, N, max(24, d // 2), 4, 6.0, 2, 100 + d), precision)


@pytest.mark.parametrize("rank,oversample", [(0, 0), (1, 1), (8, 3), (12, 8), (13, 8), (24, 8)])
@pytest.mark.parametrize("precision", [0, 1, 2])
def test_ritz_ranks(B, rank, oversample, precision):
    """Odd and even l, the largest l, and both register layouts of the preconditioner's columns."""
    check(B, layered(150, 6, 60, 4, 5.0, 3, 7), precision, ritz_rank=rank, oversample=oversample)


@pytest.mark.parametrize("columns", [2, 8])
def test_row_blocks_of_disjoint_supports(B, columns):
    """Observed columns of a 2-D grid out of each other's reach: eight consecutive observations have eight (or
    four times two) different sets of neighbours; with eight columns their union is beyond the blocks' capacity."""
    nx, ny = 50 * columns, 40
    grid = workloads.Grid((nx, ny, 1), (True, True, False), (0.4, 3.0, 1.0), True)
    pr = workloads.random_obs_problem(grid, N=5, d=ny * columns, r2=0.8, Q=2, tol=1e-6, seed=11)
    obs = (np.arange(ny)[:, None] * nx + 50 * np.arange(columns)[None, :]).reshape(-1).astype(np.int64)
    check(B, dataclasses.replace(pr, obs_idx=obs, y=pr.truth[obs] + 0.5), 1)


@pytest.mark.parametrize("precision", [0, 1])
def test_equal_eigenvalues(B, precision):
    """Observations out of each other's reach with equal variances: C is a multiple of the identity."""
    n, N = 240, 6
    rng = np.random.default_rng(3)
    base = rng.standard_normal(N)
    base -= base.mean()
    X = np.stack([np.roll(base, int(s)) for s in rng.integers(0, N, n)], axis=1)
    obs = np.arange(0, n, 12)
    R = np.full(obs.size, 0.5)
    grid = workloads.Grid((n, 1, 1), (True, False, False), (5.0, 1.0, 1.0), True)
    y = X[0, obs] + 0.5
    check(B, workloads.Problem("equal", grid, X, X[0], obs, y, R, 3, 1e-6), precision)


@pytest.mark.parametrize("n,d,N,precision", [(203, 1, 3, 0), (203, 20, 33, 0), (64, 64, 40, 1), (6400, 5, 3, 0),
                                             (6401, 5, 3, 0)])
def test_weighted_sums_sizes(B, n, d, N, precision):
    """Ragged blocks of four grid points, more members than a warp, and both sides of the grid size whose rows of
    the localized covariance fit shared memory."""
    tol, bound = BOUND[precision]
    pr = workloads.gaussian_problem_1d("sums", n=n, N=N, length_scale=4.0, obs_stride=max(1, n // d), r2=0.5,
                                       half_width=9.0, Q=2, tol=tol, seed=n + d)
    H, (rowptr, col, val) = workloads.gaussian_channel_operator(n, d, 3.0)
    R = np.full(d, 0.5)
    y = H @ pr.truth + 0.3
    outs, stats = B.info_esrf_analysis_batched(
        [dict(grid=pr.grid, X=dev(pr.X), H=(dev(rowptr), dev(col), dev(val)), y=dev(y), R=dev(R), Q=pr.Q, tol=tol)],
        B.make_options(precision=precision))
    torch.cuda.synchronize()
    assert stats[0]["status"] == 0, stats
    A_ref = F.perturbation_update_H(pr.X, H, R, pr.grid, pr.Q)
    mu_ref = F.mean_update_H(pr.X, H, y, R, pr.grid)
    assert increment_error(outs[0][1], A_ref, pr.X - pr.X.mean(0)) <= bound
    assert mean_error(outs[0][0], mu_ref, pr.X.mean(0)) <= bound
