"""AdjointEnergy takes theta in every floating type torch trains in, and integers: the energy and the
gradient are those of the same angles in float64 (bit for bit: the angles convert exactly), the gradient
arrives in theta's own type."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name", ["float64", "float32", "float16", "bfloat16", "int64"])
@pytest.mark.parametrize("shape", [(24,), (4, 6)])
def test_theta_types(name, shape):
    import torch

    from paper_2411_18354_gb300.autograd import AdjointEnergy

    gates = W.hea_circuit(4, 3)
    dt = getattr(torch, name)
    theta = torch.tensor(np.random.default_rng(2).uniform(-3, 3, shape), device="cuda").to(dt)
    exact = theta.double().reshape(-1).requires_grad_()
    want = AdjointEnergy.apply(exact, 4, gates, "c128")
    want.backward()
    if len(shape) == 1 and dt.is_floating_point:
        theta.requires_grad_()
    got = AdjointEnergy.apply(theta, 4, gates, "c128")
    assert got.dtype == torch.float64 and got.item() == want.item()
    if theta.requires_grad:
        got.backward()
        assert theta.grad.dtype == dt
        assert torch.equal(theta.grad, exact.grad.to(dt))
