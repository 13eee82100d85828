"""The autotuner times every candidate that the workspace it was given can run."""
import ctypes

import numpy as np
import pytest
import torch

from paper_2503_00253_gb300 import workloads

pytestmark = pytest.mark.gpu


def dev(a):
    return torch.tensor(np.ascontiguousarray(a), device="cuda")


@pytest.mark.parametrize("precision", [0, 1])
def test_every_candidate_that_fits_is_timed(precision):
    """Launches of the autotuner against those of its candidates: each runs once and is timed five times."""
    from paper_2503_00253_gb300 import binding as B
    pr = workloads.gaussian_problem_1d("tune", n=2048, N=8, length_scale=16.0, obs_stride=4, r2=0.5, half_width=64.0,
                                       Q=4, tol=1e-6, seed=5)
    X, obs, y, R = (dev(a) for a in (pr.X, pr.obs_idx, pr.y, pr.R))
    ws = B.workspace(B.workspace_size(pr.grid, pr.N, pr.d, pr.Q, B.make_options(precision=precision)))
    expected = 0
    for cluster_size in (0, 4, -1):
        for power_iters in (0, 1):
            for oversample in (2, 6, 10):
                o = B.make_options(precision=precision, cluster_size=cluster_size, power_iters=power_iters,
                                   oversample=oversample)
                before = B.launch_count()
                _, _, st = B.info_esrf_analysis(pr.grid, X, obs, y, R, pr.Q, pr.tol, o, ws=ws)
                assert st["status"] == 0 and st["n_unconverged"] == 0
                expected += 6 * (B.launch_count() - before)
    opts = B.make_options(precision=precision)
    before = B.launch_count()
    assert B.autotune([dict(grid=pr.grid, X=X, obs_idx=obs, y=y, R=R, Q=pr.Q, tol=pr.tol)], opts, ws=ws) > 0.0
    assert B.launch_count() - before == expected


def test_candidates_that_do_not_fit_are_skipped():
    """A workspace below every candidate's need: no call runs, and the code stays that of no candidate."""
    from paper_2503_00253_gb300 import binding as B
    pr = workloads.gaussian_problem_1d("tune", n=512, N=8, length_scale=16.0, obs_stride=4, r2=0.5, half_width=32.0,
                                       Q=4, tol=1e-6, seed=5)
    X, obs, y, R = (dev(a) for a in (pr.X, pr.obs_idx, pr.y, pr.R))
    arr = (B.ProblemC * 1)()
    mu, A = torch.empty_like(X[0]), torch.empty_like(X)
    B._fill_problem(arr[0], dict(grid=pr.grid, obs_idx=obs, y=y, R=R, Q=pr.Q, tol=pr.tol), X, mu, A)
    o, ws, best = B.make_options(precision=1), B.workspace(4096), ctypes.c_double(0.0)
    before = B.launch_count()
    code = B.library().info_esrf_autotune(arr, 1, ctypes.byref(o), ws.data_ptr(), ws.numel(),
                                          torch.cuda.current_stream().cuda_stream, ctypes.byref(best))
    assert code == -9 and B.launch_count() == before
