"""Workspace sizes, and the BF16 path's second direction buffer, which is optional.

BF16 calls of more than 384 systems keep a second copy of the search directions.  A workspace without
room for it still serves the call, with the same bits, and a reported size is not pushed past the
32 MiB of the allocation-free entry point by it.
"""
import ctypes

import numpy as np
import pytest
import torch

from paper_2503_00253_gb300 import workloads

# (nx, ny, half-width), observations, members, nodes, bytes without the second buffer of the layout before it existed
NEAR_LIMIT = [((64, 32, 6.0), 1024, 40, 44, 33_535_232), ((48, 48, 5.0), 576, 64, 47, 33_404_672),
              ((96, 64, 5.0), 1000, 40, 42, 33_007_616)]


def grid_of(shape):
    nx, ny, hw = shape
    return workloads.Grid((nx, ny, 1), (True, True, False), (hw, hw, 1.0), True)


@pytest.mark.parametrize("shape,d,N,Q,before", NEAR_LIMIT)
def test_reported_size_stays_within_the_allocation_free_limit(shape, d, N, Q, before):
    from paper_2503_00253_gb300 import binding as B
    size = B.workspace_size(grid_of(shape), N, d, Q, B.make_options(precision=2))
    assert 0 < size <= before <= 32 << 20


# (precision, solver, problems, members, observations, nodes, rank, oversample, mean only), bytes: a program's own
# buffers of these sizes have served these calls (48 x 48 points, 160 SMs, no optional part)
SERVED = [((2, 0, 1, 8, 1, 2, 10, 10, True), 323_840), ((2, 0, 1, 8, 129, 2, 10, 0, True), 695_296),
          ((2, 0, 1, 8, 129, 2, 24, 0, True), 742_912), ((2, 0, 1, 8, 500, 2, 24, 0, False), 2_122_752),
          ((0, 0, 1, 20, 60, 16, 10, 10, False), 2_335_744), ((0, 0, 64, 3, 20, 2, 10, 10, False), 42_847_488),
          ((0, 1, 1, 20, 60, 16, 10, 10, False), 2_335_744), ((0, 1, 64, 3, 20, 2, 10, 10, False), 42_847_488),
          ((0, 2, 1, 20, 60, 16, 10, 10, False), 5_586_688), ((0, 2, 64, 3, 20, 2, 0, 0, False), 73_469_184),
          ((1, 1, 1, 20, 60, 16, 10, 10, False), 1_482_752), ((1, 1, 64, 3, 20, 2, 10, 10, False), 28_822_784),
          ((1, 2, 7, 3, 20, 2, 10, 10, True), 4_305_920)]


@pytest.mark.parametrize("form,served", SERVED)
def test_calls_need_no_more_than_they_did(form, served):
    from paper_2503_00253_gb300 import binding as B
    precision, solver, count, N, d, Q, rank, oversample, mean_only = form
    o = B.make_options(precision=precision, solver=solver, ritz_rank=rank, oversample=oversample)
    arr = (B.ProblemC * count)()
    for p in arr:
        p.grid = B.make_grid(grid_of((48, 48, 5.0)))
        p.N, p.d, p.Q, p.tol = N, d, Q, 1e-6
        p.X = p.obs_idx = p.y = p.R_diag = p.mu_a = 256   # sizes only: never read
        if not mean_only:
            p.A_a = 256
    assert 0 < B.library().info_esrf_batched_workspace_size(arr, count, ctypes.byref(o)) <= served


def test_bf16_calls_of_many_observations_need_no_more_than_they_did():
    from paper_2503_00253_gb300 import binding as B
    o = B.make_options(precision=2, ritz_rank=24, oversample=8)
    assert 0 < B.workspace_size(grid_of((96, 64, 5.0)), 16, 5000, 2, o) <= 172_187_392


def dev(a):
    return torch.tensor(np.ascontiguousarray(a), device="cuda")


def problem(shape, d, N, Q):
    return workloads.random_obs_problem(grid_of(shape), N=N, d=d, r2=0.8, Q=Q, tol=1e-6, seed=d + N)


@pytest.mark.gpu
@pytest.mark.parametrize("shape,d,N,Q", [c[:4] for c in NEAR_LIMIT])
def test_allocation_free_call_near_the_limit(shape, d, N, Q):
    from paper_2503_00253_gb300 import binding as B
    pr = problem(shape, d, N, Q)
    X, obs, y, R = (dev(a) for a in (pr.X, pr.obs_idx, pr.y, pr.R))
    o = B.make_options(precision=2)
    roomy = B.workspace(B.workspace_size(pr.grid, N, d, Q, o) + 2 * (N * Q + 1) * (d + 128) + 1024)
    mu, A, st = B.info_esrf_analysis(pr.grid, X, obs, y, R, Q, pr.tol, o, ws=roomy)
    assert st["status"] == 0
    fn = B.library().info_esrf_analysis_noalloc
    P = ctypes.POINTER
    fn.restype = ctypes.c_int32
    fn.argtypes = [P(B.Grid), ctypes.c_int64, ctypes.c_void_p, ctypes.c_int64, ctypes.c_void_p, ctypes.c_void_p,
                   ctypes.c_void_p, ctypes.c_int32, ctypes.c_double, P(B.Options), ctypes.c_void_p,
                   ctypes.c_void_p, ctypes.c_void_p]
    mu2, A2 = torch.full_like(mu, float("nan")), torch.full_like(A, float("nan"))
    rc = fn(ctypes.byref(B.make_grid(pr.grid)), N, X.data_ptr(), d, obs.data_ptr(), y.data_ptr(), R.data_ptr(), Q,
            pr.tol, ctypes.byref(o), torch.cuda.current_stream().cuda_stream, mu2.data_ptr(), A2.data_ptr())
    torch.cuda.synchronize()
    assert rc == 0
    assert torch.equal(mu, mu2) and torch.equal(A, A2)


@pytest.mark.gpu
@pytest.mark.parametrize("shape,d,N,Q", [((48, 48, 5.0), 129, 16, 25), ((48, 48, 5.0), 600, 40, 16),
                                         ((96, 64, 5.0), 1500, 80, 10)])
@pytest.mark.parametrize("max_iter", [1, 1000])
def test_one_direction_buffer_gives_the_same_bits(shape, d, N, Q, max_iter):
    """Workspaces of the reported size and just below it: two direction buffers, and one with a copy."""
    from paper_2503_00253_gb300 import binding as B
    pr = problem(shape, d, N, Q)
    args = [pr.grid, dev(pr.X), dev(pr.obs_idx), dev(pr.y), dev(pr.R), Q, pr.tol]
    o = B.make_options(precision=2, max_iter=max_iter)
    size = B.workspace_size(pr.grid, N, d, Q, o)
    two = B.info_esrf_analysis(*args, o, ws=B.workspace(size))
    one = B.info_esrf_analysis(*args, o, ws=B.workspace(size - 256))
    assert two[2]["status"] == one[2]["status"] and two[2]["iters_max"] == one[2]["iters_max"]
    assert torch.equal(two[0], one[0]) and torch.equal(two[1], one[1])


@pytest.mark.gpu
def test_fp32_vectors_beyond_shared_memory_run_in_the_scratch_they_had():
    """136 bytes a row and SM are asked for, 128 are enough (the optional last CTAs of 152 are left out); no
    blocks of rows at this size, so the bits are the same."""
    from paper_2503_00253_gb300 import binding as B
    d = 33000
    pr = workloads.gaussian_problem_1d("scratch", n=2 * d, N=3, length_scale=3.0, obs_stride=2, r2=0.5, half_width=3.0,
                                       Q=2, tol=1e-6, seed=3)
    args = [pr.grid, dev(pr.X), dev(pr.obs_idx), dev(pr.y), dev(pr.R), pr.Q, pr.tol]
    o = B.make_options(precision=1, ritz_rank=24, oversample=8, cluster_size=-1)
    size = B.workspace_size(pr.grid, pr.N, pr.d, pr.Q, o)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    full, served = (B.info_esrf_analysis(*args, o, ws=B.workspace(n)) for n in (size, size - 7 * d * sms))
    assert full[2]["status"] == 0 and full[2]["solver_path"] == 0
    assert torch.equal(full[0], served[0]) and torch.equal(full[1], served[1])
