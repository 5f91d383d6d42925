"""Surrogate gradients where the weight gradients' sums over the batch are cut into slices (one k block, fewer
blocks than slices, an uneven last slice) and at the narrowest and a wider output layer, against the FP64 MLP
rounding to BF16 where the GPU does: each element within 2^-6 of the sum of its absolute terms, as the unsliced
gradients are held to."""
import numpy as np
import pytest

from oracle import mlp
from paper_1311_4627_gb300 import heat
from paper_1311_4627_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,n_lambda", [(64, 64), (320, 128), (1088, 64)])
def test_gradients_with_sliced_sums(n, n_lambda):
    import torch

    lam = W.wavelength_grid(n_lambda)
    radii, _, cabs, off, T, E, sw = W.make_grains(lam, np.geomspace(4e-8, 1e-6, 2), ["carbonaceous"] * 2, [32, 40])
    dims = [heat.SURROGATE_INPUTS, 512, 512, 512, 512, n_lambda]
    rng = np.random.default_rng(n)
    xn = mlp.bf16_round(rng.normal(0, 1, (n, dims[0])))
    tn = rng.normal(0, 1, (n, n_lambda)).astype(np.float32)
    tn[rng.random(tn.shape) < 0.2] = np.nan
    ctx = heat.heat_create_grid(0, lam)
    try:
        heat.heat_set_grains(ctx, radii, cabs, off, T, E, sw)
        heat.heat_surrogate_init(ctx, 1, None, 3)
        flat = heat.heat_surrogate_params(ctx, 0)
        g = torch.empty(flat.size, dtype=torch.float32, device="cuda")
        X = torch.tensor(xn, dtype=torch.float32, device="cuda")
        heat.heat_surrogate_grads(ctx, 0, X, torch.from_numpy(tn).cuda(), n, g)
    finally:
        heat.heat_destroy(ctx)
    layers = mlp.unflatten(mlp.bf16_round(flat), dims)
    t64 = tn.astype(np.float64)
    _, ref = mlp.loss_and_grad(layers, xn, t64, quantize=mlp.bf16_round)
    scale = mlp.gradient_scale(layers, xn, t64, quantize=mlp.bf16_round)
    assert np.all(np.abs(g.cpu().numpy() - ref) <= 2.0**-6 * np.maximum(scale, 1e-30))
