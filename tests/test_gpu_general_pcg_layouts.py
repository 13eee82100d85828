"""The general PCG kernel on both sides of every rule that changes its layout or matvec.

Vectors of a group in 200 KB of shared memory (level 0), the direction alone (1) or none (2), for
FP32 groups of eight systems, FP64 groups of one (up to two systems per SM) and of two; C by blocks
of four rows, its overflow, and C by rows.  Reference: block CG in FP64, a kernel and an algorithm of its
own on the same covariances, at tolerance 1e-12 (small sizes are compared with the oracle elsewhere).
Bounds of the end-to-end parity tests: 1e-10 at tolerance 1e-12 (FP64), 1e-4 at 1e-6 (FP32).
"""
import dataclasses

import numpy as np
import pytest
import torch

from oracle import filter as F
from paper_2503_00253_gb300 import workloads
from parity_checks import increment_error, mean_error

pytestmark = pytest.mark.gpu

TOL, BOUND = {0: 1e-12, 1: 1e-6}, {0: 1e-10, 1: 1e-4}


@pytest.fixture(scope="module")
def B():
    from paper_2503_00253_gb300 import binding
    binding.library()
    return binding


def dev(a):
    return torch.tensor(np.ascontiguousarray(a), device="cuda")


def problem(d, N, Q, seed):
    grid = workloads.Grid((max(24, d // 2), 1, 4), (True, False, False), (6.0, 1.0, 1.5), True)
    return workloads.random_obs_problem(grid, N=N, d=d, r2=0.8, Q=Q, tol=1e-6, seed=seed)


def analysis(B, pr, precision, ws=None, tol=None, **kw):
    opts = B.make_options(precision=precision, **kw)
    mu_a, A_a, st = B.info_esrf_analysis(pr.grid, dev(pr.X), dev(pr.obs_idx), dev(pr.y), dev(pr.R), pr.Q,
                                         tol or TOL[precision], opts, ws=ws)
    torch.cuda.synchronize()
    assert st["status"] == 0 and st["n_unconverged"] == 0, st
    return mu_a, A_a, st


def compare(pr, got, want, bound):
    assert increment_error(got[1], want[1], pr.X - pr.X.mean(0)) <= bound
    assert mean_error(got[0], want[0], pr.X.mean(0)) <= bound


def status_words(B, pr, opts, ws):
    """The device status words that the last analysis left in its workspace."""
    p = object.__new__(B.Prepared)
    p.g, p.N, p.n, p.d, p.Q, p.o = B.make_grid(pr.grid), pr.N, pr.n, pr.d, pr.Q, opts
    p.precision, p.ws, p.stream = opts.precision, ws, None
    return p.export("status")


# FP32: level 0 up to 1505 rows, 1 up to 4298; FP64 groups of one: 6399 and 24573; of two: 3199 and 11773
@pytest.mark.parametrize("d,N,Q,precision", [
    (1505, 3, 2, 1), (1506, 3, 2, 1), (4298, 3, 2, 1), (4299, 3, 2, 1), (2050, 9, 3, 1), (2051, 9, 3, 1),
    (6399, 3, 2, 0), (6400, 3, 2, 0), (24573, 3, 2, 0), (24574, 3, 2, 0),
    (3199, 20, 16, 0), (3200, 20, 16, 0), (11773, 20, 16, 0), (11774, 21, 16, 0)])
def test_levels(B, d, N, Q, precision):
    pr = problem(d, N, Q, d)
    got = analysis(B, pr, precision)
    assert got[2]["solver_path"] == 0
    compare(pr, got, analysis(B, pr, 0, solver=B.SOLVER_BLOCK), BOUND[precision])


def columns(count):
    """Observed columns of a 2-D grid out of each other's reach, 13 neighbours per observation: four consecutive
    observations see up to 52 different ones."""
    nx, ny = 50 * count, 40
    grid = workloads.Grid((nx, ny, 1), (True, True, False), (0.4, 3.0, 1.0), True)
    pr = workloads.random_obs_problem(grid, N=5, d=ny * count, r2=0.8, Q=2, tol=1e-6, seed=11)
    obs = (np.arange(ny)[:, None] * nx + 50 * np.arange(count)[None, :]).reshape(-1).astype(np.int64)
    return dataclasses.replace(pr, obs_idx=obs, y=pr.truth[obs] + 0.5)


@pytest.mark.parametrize("count,overflow", [(1, 0), (2, 0), (4, 1), (8, 1)])
def test_union_of_four_rows_beyond_the_capacity(B, count, overflow):
    """With 13 neighbours per row a block holds 34 columns: one and two columns fit (16 and 28), four and eight
    (52) don't, and the matvec goes by rows."""
    pr = columns(count)
    opts = B.make_options(precision=1, max_neighbors=13)
    ws = B.workspace(B.workspace_size(pr.grid, pr.N, pr.d, pr.Q, opts))
    got = analysis(B, pr, 1, ws=ws, max_neighbors=13)
    assert list(status_words(B, pr, opts, ws)[[0, 2]]) == [0, overflow]
    compare(pr, got, (F.mean_update(pr.X, pr.obs_idx, pr.y, pr.R, pr.grid),
                      F.perturbation_update(pr.X, pr.obs_idx, pr.R, pr.grid, pr.Q)), BOUND[1])


@pytest.mark.parametrize("d", [1, 6, 127, 130, 514, 1506])
def test_without_the_blocks_of_rows(B, d):
    """A workspace that holds everything but the blocks of four rows."""
    pr = problem(d, 5, 2, d)
    size = B.workspace_size(pr.grid, pr.N, pr.d, pr.Q, B.make_options(precision=1))
    want = (F.mean_update(pr.X, pr.obs_idx, pr.y, pr.R, pr.grid),
            F.perturbation_update(pr.X, pr.obs_idx, pr.R, pr.grid, pr.Q))
    compare(pr, analysis(B, pr, 1, ws=B.workspace(size - 1)), want, BOUND[1])
