"""The matrix build in two passes (photon prefixes, then pieces of the elements) against the one-walk
build that the no-allocation entry point runs: the same B, so the same P bit for bit, at sizes that
leave ragged ends: a last group of one cell, an odd group for the two-group warps, an odd grain for
the two-grain walks, more groups than one block takes, grids of few segments (long pieces of one
segment) and of more segments than entries."""
import numpy as np
import pytest

from paper_1311_4627_gb300 import heat
from paper_1311_4627_gb300 import workloads as W
from tests.gpu_helpers import Lib

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("build", [heat.HEAT_BUILD_F32, heat.HEAT_BUILD_F64])
@pytest.mark.parametrize("cells,grains,n_lambda", [(17, 1, 2), (33, 3, 3), (64, 2, 40), (97, 5, 257), (545, 1, 1100)])
def test_two_passes_equal_one_walk(build, cells, grains, n_lambda):
    import torch

    lam = W.wavelength_grid(n_lambda)
    radii = np.geomspace(4e-8, 3e-5, grains)
    comps = ["carbonaceous", "silicate"] * 3
    rng = np.random.Generator(np.random.PCG64(cells))
    u = W.three_bb_fields(lam, 10.0 ** rng.uniform(-2, 4, cells), rng.uniform(-1, 1, cells),
                          10.0 ** rng.uniform(-2, 0, (cells, 3)))
    u[-1] = 0.0  # a cell without field
    u[0, : n_lambda // 3] = 0.0  # inactive segments
    wl = W.custom(lam, radii, comps[:grains], [33 + 40 * g for g in range(grains)], u)
    lib = Lib(wl)
    try:
        lib.set_fields(wl.u)
        P, _ = lib.solve(want_j=False, build=build)
        P1 = torch.empty(cells, wl.total_bins, dtype=torch.float64, device="cuda")
        heat.heat_solve_noalloc(lib.ctx, build, lib.u, cells, P1)
        heat.heat_sync(lib.ctx)
        assert np.array_equal(P, P1.cpu().numpy())
    finally:
        lib.close()
