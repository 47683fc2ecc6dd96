"""ring_chi2's place in autograd, without a GPU (a context that answers with
fixed numbers): theta is its only differentiable input, whatever the other
arguments require."""
import numpy as np
import pytest

from paper_2309_12496_gb300 import rich

torch = pytest.importorskip("torch")

GRAD = np.arange(1.0, 11.0)


class FixedContext:
    def trace_grad(self, tracks, theta, targets, outputs, sigma=1.0, seed=0):
        return 3.5 * float(sigma), GRAD.copy(), 7


@pytest.mark.parametrize("theta_grad", [False, True])
@pytest.mark.parametrize("target_grad", [False, True])
def test_only_theta_is_differentiated(theta_grad, target_grad):
    theta = torch.zeros(10, dtype=torch.float64, requires_grad=theta_grad)
    targets = torch.zeros(4, requires_grad=target_grad)
    sigma = torch.tensor(2.0, requires_grad=target_grad)
    loss = rich.ring_chi2(FixedContext(), theta, None, targets, None, sigma=sigma, seed=1)
    assert loss.item() == 7.0 and loss.requires_grad == theta_grad
    if theta_grad:
        assert loss.grad_fn.n_used == 7
        (2.0 * loss).backward()
        np.testing.assert_array_equal(theta.grad.numpy(), 2.0 * GRAD)
        assert targets.grad is None
