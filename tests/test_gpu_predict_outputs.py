"""Ensemble statistics with 16-byte accesses against the scalar ones: the same samples into an aligned output and into one
that is only 4-byte aligned, the same bits."""
import numpy as np
import pytest

from paper_1311_4627_gb300 import heat
from paper_1311_4627_gb300 import workloads as W
from tests.gpu_helpers import Lib

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("members", [2, 5])
@pytest.mark.parametrize("n_lambda", [64, 192])
def test_aligned_and_unaligned_outputs_agree(members, n_lambda):
    import torch

    lam = W.wavelength_grid(n_lambda)
    rng = np.random.Generator(np.random.PCG64(members))
    u = W.three_bb_fields(lam, 10.0 ** rng.uniform(-1, 2, 24), rng.uniform(-1, 1, 24), 10.0 ** rng.uniform(-1, 0, (24, 3)))
    wl = W.custom(lam, np.array([1e-6, 3e-6]), ["carbonaceous", "silicate"], [64, 64], u)
    lib = Lib(wl)
    try:
        lib.set_fields(wl.u)
        _, j = lib.solve(want_P=False, j_dtype=heat.HEAT_F32, build=heat.HEAT_BUILD_F64)
        n = 24 * 2
        jd = torch.from_numpy(j.astype(np.float32)).cuda().reshape(n, n_lambda)
        heat.heat_surrogate_init(lib.ctx, members, np.zeros(2), seed=1)
        X = torch.empty(n, heat.SURROGATE_INPUTS, device="cuda")
        Y = torch.empty(n, n_lambda, device="cuda")
        lnp = torch.empty(n, device="cuda")
        st = torch.cuda.current_stream().cuda_stream
        heat.heat_surrogate_samples(lib.ctx, 0, 24, jd, X, Y, lnp, st)
        heat.heat_surrogate_fit_norm(lib.ctx, X, Y, n, st)
        a = torch.empty(n, n_lambda, device="cuda")
        sa = torch.empty(n, device="cuda")
        heat.heat_surrogate_predict(lib.ctx, X, lnp, n, a, sa, st)
        buf = torch.empty(n * n_lambda + 1, device="cuda")
        sb = torch.empty(n, device="cuda")
        heat.heat_surrogate_predict(lib.ctx, X, lnp, n, buf[1:], sb, st)  # 4-byte aligned only
        torch.cuda.synchronize()
        assert torch.equal(a.reshape(-1).view(torch.int32), buf[1:].clone().view(torch.int32))
        assert torch.equal(sa.view(torch.int32), sb.view(torch.int32))
    finally:
        lib.close()
