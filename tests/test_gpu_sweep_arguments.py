"""Batch.feed_forward_vjp refuses tensors that its kernels would read or write
out of bounds: a theta_bar that does not hold the network's parameters on the
device, steps that are not one after another in memory."""
import pytest
import torch

from paper_2203_13760_gb300 import inputs, jf

pytestmark = pytest.mark.gpu


def test_bad_theta_bar_and_steps_are_refused():
    theta = torch.tensor(inputs.nn_params(), dtype=torch.float32, device="cuda")
    b = jf.Batch([jf.make_grid((16, 12), bc=(1,) * 6)] * 2, dtype="f32", flux="rusanov-nn", integrator="rk2", nn=theta)
    U = [torch.tensor(inputs.random_smooth((16, 12), seed=k).U, dtype=torch.float32, device="cuda") for k in (1, 2)]
    trajs = b.feed_forward(U, 2, 1e-4)
    grads = [torch.ones_like(t) for t in trajs]
    dt = torch.full((2,), 1e-4, dtype=torch.float64, device="cuda")
    good = torch.zeros_like(theta)
    for bad in (good[:-1], good.double(), good.cpu(), torch.zeros(2 * theta.numel(), device="cuda")[::2]):
        with pytest.raises(ValueError, match="theta_bar"):
            b.feed_forward_vjp(trajs, grads, 2, dt, bad)
    with pytest.raises(ValueError, match="dt"):
        b.feed_forward_vjp(trajs, grads, 2, torch.full((4,), 1e-4, dtype=torch.float64, device="cuda")[::2], good)
    lam = b.feed_forward_vjp(trajs, grads, 2, dt, good)
    assert all(torch.isfinite(x).all() for x in lam) and bool(good.any())
