"""The recursion with a block of four warps per task against the one with a warp per task (the no-allocation entry point
takes a warp per task): the same bits, at row counts around multiples of the block's four rows, bands narrower and wider
than a block, with spectra that pass the overflow guard, and with tail pruning against the few-cell kernel."""
import numpy as np
import pytest

from paper_1311_4627_gb300 import heat
from paper_1311_4627_gb300 import workloads as W
from tests.gpu_helpers import Lib

pytestmark = pytest.mark.gpu


def _case(bins, cells, seed, hot=False):
    rng = np.random.Generator(np.random.PCG64(seed))
    lam = W.wavelength_grid(96)
    u = W.three_bb_fields(lam, 10.0 ** rng.uniform(-2, 4, cells), rng.uniform(-1, 1, cells),
                          10.0 ** rng.uniform(-2, 0, (cells, 3)))
    if hot:
        u *= 10.0 ** rng.uniform(0, 12, (cells, 1))  # X grows past 2^800: rescales
    radii = np.geomspace(3.5e-8, 1e-5, len(bins))
    return W.custom(lam, radii, ["carbonaceous", "silicate"] * 8, list(bins), u)


@pytest.mark.parametrize("build", [heat.HEAT_BUILD_F32, heat.HEAT_BUILD_F64])
@pytest.mark.parametrize("bins,hot", [((2, 3, 4, 5, 6, 7, 8, 9), False), ((33, 34, 35, 36, 37), False),
                                      ((97, 130, 255), False), ((130, 255, 514), True)])
def test_block_tasks_equal_warp_tasks(build, bins, hot):
    import torch

    wl = _case(bins, 50, len(bins), hot)
    lib = Lib(wl)
    try:
        lib.set_fields(wl.u)
        P, _ = lib.solve(want_j=False, build=build)
        P1 = torch.empty(wl.n_cells, wl.total_bins, dtype=torch.float64, device="cuda")
        heat.heat_solve_noalloc(lib.ctx, build, lib.u, wl.n_cells, P1)
        heat.heat_sync(lib.ctx)
        assert np.array_equal(P, P1.cpu().numpy())
        assert np.all(np.isfinite(P)) and np.allclose(P[:, :bins[0]].sum(axis=1), 1.0)
    finally:
        lib.close()


@pytest.mark.parametrize("bins", [(33, 34, 35, 36), (255, 514)])
def test_block_tasks_prune_as_the_few_cell_kernel(bins):
    """Tail pruning drops shares below 2^-L of the total: 1e-9 of the probability and of each row's largest."""
    wl = _case(bins, 50, 7)
    lib = Lib(wl)
    try:
        lib.set_fields(wl.u)
        P, _ = lib.solve(want_j=False, build=heat.HEAT_BUILD_F64, prune_eps=1e-9)
        lib.set_fields(wl.u[:3])
        Q, _ = lib.solve(want_j=False, build=heat.HEAT_BUILD_F64, prune_eps=1e-9)
        assert np.array_equal(P[:3] == 0.0, Q == 0.0)
        assert np.all(np.abs(P[:3] - Q) <= 1e-10 * Q)
    finally:
        lib.close()
