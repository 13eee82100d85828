"""Loss and gradient of the training step at the sizes where its kernels change their way of
working, against the FP64 oracle.

e sums 2 x 17 products in FP32: 34 roundings of 2^-24 on terms a few times larger than e, so
1e-5 of the gradient's norm; 1e-4 is asked for.
"""
import numpy as np
import pytest
import torch

from oracle import learned as LR

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    from paper_2503_00253_gb300 import binding
    binding.library()
    return binding


def dev(a):
    return torch.tensor(np.ascontiguousarray(a), device="cuda")


# fewer observations than the stencil's taps, rows that are no multiple of four, one row more than a block's 512,
# the largest, more samples than resident blocks
@pytest.mark.parametrize("d,S", [(1, 2), (3, 2), (16, 3), (17, 3), (33, 2), (512, 2), (513, 2), (1030, 2), (8533, 1),
                                 (20, 700)])
def test_training_step_sizes(B, d, S):
    rng = np.random.default_rng(d)
    theta = LR.init_params(seed=1, scale=0.3).astype(np.float32)
    phi = LR.features(np.exp(rng.uniform(0.1, 6.0, S)), 2.0, 140.0).astype(np.float32)
    V, Y, Z = (rng.standard_normal((S, d)).astype(np.float32) for _ in range(3))
    loss, grad = B.learn_loss_grad(dev(theta), dev(phi), dev(V), dev(Y), dev(Z))
    args = [a.astype(np.float64) for a in (phi, V, Y, Z)]
    t = theta.astype(np.float64)
    assert abs(loss - LR.loss(t, *args)) < 1e-5 * loss
    g = grad.cpu().numpy().astype(np.float64)
    for _ in range(3):   # directional derivatives by central differences (error of order 1e-8)
        u = rng.standard_normal(t.size)
        u *= np.linalg.norm(g) / np.linalg.norm(u)
        u = (u + g) / np.linalg.norm(u + g)
        fd = (LR.loss(t + 1e-5 * u, *args) - LR.loss(t - 1e-5 * u, *args)) / 2e-5
        assert abs(g @ u - fd) < 1e-4 * np.linalg.norm(g)


def test_training_step_takes_rows_off_16_byte_boundaries(B):
    rng = np.random.default_rng(2)
    d, S = 64, 4
    theta = dev(LR.init_params(seed=1, scale=0.3).astype(np.float32))
    phi = dev(LR.features(np.array([1.1, 3.0, 20.0, 300.0]), 2.0, 140.0).astype(np.float32))
    flat = [dev(rng.standard_normal(S * d + 1).astype(np.float32)) for _ in range(3)]
    off = [f[1:].view(S, d) for f in flat]
    l0, g0 = B.learn_loss_grad(theta, phi, *off)
    l1, g1 = B.learn_loss_grad(theta, phi, *(o.clone() for o in off))
    assert l0 == l1 and torch.equal(g0, g1)
