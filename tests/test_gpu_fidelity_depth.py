"""The deepest circuits whose fidelity one CTA serves: 16 bytes of shared memory per
angle and amplitude beside 128 bytes of the reduction's.

n = 1: all rotations are about one axis, the state is the one of the summed angle
(the sum of 14,518 angles below 1e-3 and as many rotations: 1e-10)."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("less", [0, 1, 3, 1000])
def test_deepest_circuit(dv, ctx, less):
    optin = torch.cuda.get_device_properties(0).shared_memory_per_block_optin
    P = (optin - 128) // 16 - 2 - less
    alpha = np.random.default_rng(less).uniform(-1e-3, 1e-3, P)
    x = np.array([0.6, 0.0, 0.8, 0.0])  # (0.6, 0.8), complex
    F = np.zeros(1)
    dv.dvqls_fidelity(ctx, dv.make_ansatz(1, P - 1), alpha, x, F)
    h = alpha.sum() / 2
    assert abs(F[0] - (0.6 * np.cos(h) + 0.8 * np.sin(h)) ** 2) <= 1e-10
