"""The surrogate's loss over batches of which a thread takes many entries: summed without the drift of a long FP32 sum."""
import numpy as np
import pytest

from paper_1311_4627_gb300 import heat
from paper_1311_4627_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [64, 8192, 16384])
def test_loss_of_equal_errors(n):
    """Targets that dwarf the outputs, so that every squared error is the same FP32 number and 1 / count a power of two: the
    loss is that number, to the FP64 sum's rounding."""
    import torch

    lam = W.wavelength_grid(1024)
    radii, _, cabs, off, T, E, sw = W.make_grains(lam, np.geomspace(4e-8, 1e-6, 2), ["carbonaceous"] * 2, [32, 40])
    value = np.float32(1.2345678e9)  # a unit in its last place is 128
    ctx = heat.heat_create_grid(0, lam)
    try:
        heat.heat_set_grains(ctx, radii, cabs, off, T, E, sw)
        heat.heat_surrogate_init(ctx, 1, None, 3)
        g = torch.empty(heat.heat_surrogate_params(ctx, 0).size, dtype=torch.float32, device="cuda")
        X = torch.zeros(n, heat.SURROGATE_INPUTS, device="cuda")
        loss = heat.heat_surrogate_grads(ctx, 0, X, torch.full((n, 1024), float(value), device="cuda"), n, g)
    finally:
        heat.heat_destroy(ctx)
    assert abs(loss / float(value * value) - 1.0) <= 1e-12


def test_loss_that_overflows():
    """Squared errors beyond FP32: an infinite loss, not a NaN."""
    import torch

    lam = W.wavelength_grid(64)
    radii, _, cabs, off, T, E, sw = W.make_grains(lam, np.geomspace(4e-8, 1e-6, 2), ["carbonaceous"] * 2, [32, 40])
    ctx = heat.heat_create_grid(0, lam)
    try:
        heat.heat_set_grains(ctx, radii, cabs, off, T, E, sw)
        heat.heat_surrogate_init(ctx, 1, None, 3)
        g = torch.empty(heat.heat_surrogate_params(ctx, 0).size, dtype=torch.float32, device="cuda")
        X = torch.zeros(64, heat.SURROGATE_INPUTS, device="cuda")
        loss = heat.heat_surrogate_grads(ctx, 0, X, torch.full((64, 64), 1e20, device="cuda"), 64, g)
    finally:
        heat.heat_destroy(ctx)
    assert loss == np.inf
