"""The BF16 path waits for its own stream only.

Its loop reads the count of running systems on the host.  Work that the same thread has queued on
another stream (and what that work has put on the thread's side stream) must not be waited for: it
may depend on something the caller does after this call.
"""
import numpy as np
import pytest
import torch

from paper_2503_00253_gb300 import workloads

pytestmark = pytest.mark.gpu


def dev(a):
    return torch.tensor(np.ascontiguousarray(a), device="cuda")


@pytest.mark.parametrize("solver", [0, 1])
def test_bf16_call_does_not_wait_for_other_streams(solver):
    from paper_2503_00253_gb300 import binding as B
    p1 = workloads.gaussian_problem_1d("other", n=512, N=8, length_scale=8.0, obs_stride=4, r2=0.5, half_width=16.0,
                                       Q=4, tol=1e-6, seed=1)
    p2 = workloads.gaussian_problem_2d(nx=48, ny=48, N=8, length_scale=6.0, obs_stride=2, r2=0.5, half_width=6.0,
                                       Q=4, tol=1e-6, seed=2)
    args1, args2 = ([p.grid, dev(p.X), dev(p.obs_idx), dev(p.y), dev(p.R), p.Q, p.tol] for p in (p1, p2))
    o1, o2 = B.make_options(precision=1, solver=solver), B.make_options(precision=2)
    ref1, ref2 = (B.info_esrf_analysis(*a, o)[:2] for a, o in ((args1, o1), (args2, o2)))   # first calls, lazy loading
    ws1 = B.workspace(B.workspace_size(p1.grid, p1.N, p1.d, p1.Q, o1))
    ws2 = B.workspace(B.workspace_size(p2.grid, p2.N, p2.d, p2.Q, o2))
    out1, out2 = ([torch.zeros_like(t) for t in r] for r in (ref1, ref2))
    torch.cuda.synchronize()
    a, b, done = torch.cuda.Stream(), torch.cuda.Stream(), torch.cuda.Event()
    with torch.cuda.stream(a):
        torch.cuda._sleep(3_000_000_000)   # about 1.5 s
    B.info_esrf_analysis(*args1, o1, ws=ws1, mu_a=out1[0], A_a=out1[1], stats=False, stream=a)
    done.record(a)
    B.info_esrf_analysis(*args2, o2, ws=ws2, mu_a=out2[0], A_a=out2[1], stats=False, stream=b)
    waited = done.query()
    torch.cuda.synchronize()
    assert not waited
    assert torch.equal(out2[0], ref2[0]) and torch.equal(out2[1], ref2[1])
    assert torch.allclose(out1[0], ref1[0]) and torch.allclose(out1[1], ref1[1])
