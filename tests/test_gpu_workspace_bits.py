"""FP32 analyses give the same bits in any workspace of at least the reported size."""
import numpy as np
import pytest
import torch

from paper_2503_00253_gb300 import workloads

pytestmark = pytest.mark.gpu


def dev(a):
    return torch.tensor(np.ascontiguousarray(a), device="cuda")


def at_the_limit(B, d, N, Q):
    """The grid at which the blocks of C leave the reported size, which they alone would push past 32 MiB."""
    last = 0
    for nx in range(d, 9000, 8):
        grid = workloads.Grid((nx, 1, 4), (True, False, False), (6.0, 1.0, 1.5), True)
        size = B.workspace_size(grid, N, d, Q, B.make_options(precision=1))
        if size < last:
            assert size <= 32 << 20 < size + 20 * d * d
            return grid, size
        last = size
    raise AssertionError("no such grid")


@pytest.mark.parametrize("d,N,Q", [(150, 8, 4), (500, 8, 4)])
def test_larger_workspace_gives_the_same_bits(d, N, Q):
    from paper_2503_00253_gb300 import binding as B
    grid, size = at_the_limit(B, d, N, Q)
    pr = workloads.random_obs_problem(grid, N=N, d=d, r2=0.8, Q=Q, tol=1e-6, seed=d)
    args = [pr.grid, dev(pr.X), dev(pr.obs_idx), dev(pr.y), dev(pr.R), Q, pr.tol]
    o = B.make_options(precision=1)
    exact, larger = (B.info_esrf_analysis(*args, o, ws=B.workspace(n)) for n in (size, size + (16 << 20)))
    assert exact[2]["status"] == 0 and exact[2]["solver_path"] == 0
    assert torch.equal(exact[0], larger[0]) and torch.equal(exact[1], larger[1])
