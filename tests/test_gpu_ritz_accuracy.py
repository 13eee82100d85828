"""FP64 Ritz pairs of close eigenvalues, to FP64 accuracy.

Observations out of each other's reach make C diagonal, with variances of the observation errors
chosen so that its entries are the wanted spectrum; with as many test vectors as observations the
Ritz pairs are then eigenpairs of C.

Bound: the FP64 work is at most 30 sweeps of 31 rounds that each round an entry a few times
(930 x 3 x 2^-53 = 3e-13) and a CholeskyQR factor of float-float entries (32 x 2^-47 = 2e-13).
"""
import numpy as np
import pytest
import torch

from paper_2503_00253_gb300 import workloads

pytestmark = pytest.mark.gpu

BOUND = 5e-13


@pytest.mark.parametrize("l", [7, 20, 32])
@pytest.mark.parametrize("step", [0.0, 1e-8, 1e-5, 1e-4, 1e-3, 1e-1])
def test_close_eigenvalues_keep_fp64_accuracy(l, step):
    from paper_2503_00253_gb300 import binding as B
    k = min(24, l - 3)
    rng = np.random.default_rng(l)
    grid = workloads.Grid((8 * l, 1, 1), (True, False, False), (2.0, 1.0, 1.0), True)
    X = rng.standard_normal((12, 8 * l))
    obs = np.arange(0, 8 * l, 8)
    lam = 1.0 + step * np.arange(l)
    R = X[:, obs].var(axis=0, ddof=1) / lam
    P = B.Prepared(grid, *(torch.tensor(a, device="cuda") for a in (X, obs, R)), 2,
                   B.make_options(precision=0, ritz_rank=k, oversample=l - k))
    theta = P.export("theta")
    Phi, CPhi = P.export("phi").reshape(l, k), P.export("cphi").reshape(l, k)
    assert P.export("status")[0] == 0
    top = lam.max()
    assert np.abs(theta - np.sort(lam)[::-1][:k]).max() <= BOUND * top
    assert np.abs(Phi.T @ Phi - np.eye(k)).max() <= BOUND
    assert np.abs(lam[:, None] * Phi - CPhi).max() <= BOUND * top
    assert np.abs(CPhi - Phi * theta).max() <= BOUND * top
