"""The convolutions read packed copies of the weights, which every optimiser
step rewrites: after some steps the network's loss and gradient are those of a
fresh network given the same parameters."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,n,steps", [(4, 8, 1), (5, 6, 7)])
def test_packed_weights_follow_the_optimiser(L, n, steps):
    from paper_2412_01737_gb300 import Net
    rng = np.random.default_rng(L)
    th = rng.uniform(0, 2 * np.pi, (n, 2 * L * L))
    bl = rng.integers(0, L, (n, 2))
    net = Net(0, L, 3)
    before = net.get_params()
    g0 = net.loss_grad(th, bl)[1]
    net.train(torch.as_tensor(th, device="cuda"), n, steps, 1e-2)
    params = net.get_params()
    fresh = Net(0, L, 3)
    fresh.set_params(params)
    (la, ga), (lb, gb) = net.loss_grad(th, bl), fresh.loss_grad(th, bl)
    net.close()
    fresh.close()
    # every step moves each weight by up to lr: stale weights of any layer and
    # direction would show in the gradient at the size of this change
    assert np.abs(params - before).max() > 5e-3
    assert np.linalg.norm(ga - g0) > 1e-2 * np.linalg.norm(g0)
    assert abs(la - lb) <= 1e-6 * abs(lb)
    assert np.linalg.norm(ga - gb) <= 1e-6 * np.linalg.norm(gb)
