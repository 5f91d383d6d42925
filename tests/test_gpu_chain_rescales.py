"""The recursion where spectra pass the overflow guard, against the FP64 oracle.  Few cells: in every run of eight columns,
in some of them, and in the last, partial one; one warp, four and six warps per spectrum.  Many cells: by a warp and by a
block of four warps per task."""
import numpy as np
import pytest

import oracle
from paper_1311_4627_gb300 import heat
from paper_1311_4627_gb300 import workloads as W

from .gpu_helpers import Lib, relerr

pytestmark = pytest.mark.gpu


def _workload(bins, cells, scale):
    rng = np.random.default_rng(cells)
    lam = W.wavelength_grid(96)
    u = W.three_bb_fields(lam, 10.0 ** rng.uniform(0, 2, cells), rng.uniform(-1, 1, cells),
                          10.0 ** rng.uniform(-2, 0, (cells, 3))) * 10.0 ** scale
    return W.custom(lam, np.geomspace(3.5e-8, 1e-6, len(bins)), ["carbonaceous", "silicate"] * 2, list(bins), u)


# fields so strong that X grows by 2^400 to 2^1000 in eight states (the guard is at 2^800); the exact path's 1e-10
@pytest.mark.parametrize("scale", [25, 35, 45])
@pytest.mark.parametrize("bins", [(7, 8, 9, 17), (37, 100, 161)])
@pytest.mark.parametrize("cells", [1, 3])
def test_rescales_in_consecutive_runs(scale, bins, cells):
    wl = _workload(bins, cells, scale)
    P_ref, _, _, st = oracle.solve_batch(wl, oracle.grain_cooling(wl), want_j=False)
    assert st == oracle.OK
    if scale == 45:
        top = P_ref[0, wl.grain_slice(len(bins) - 1)]
        assert top[-9] < 2.0 ** -850 * top[-1]  # a rescale in each of the last runs
    lib = Lib(wl)
    try:
        lib.set_fields(wl.u)
        first, _ = lib.solve(want_j=False, build=heat.HEAT_BUILD_F64)
        r, ok = relerr(first, P_ref)
        assert ok and r <= 1e-10, r
        for _ in range(20):
            P, _ = lib.solve(want_j=False, build=heat.HEAT_BUILD_F64)
            assert np.array_equal(P, first)
    finally:
        lib.close()


# 20 cells: heat_solve gives the wide grains of so short a launch a block per task, the no-allocation entry point a warp
@pytest.mark.parametrize("scale", [25, 35, 45])
@pytest.mark.parametrize("bins", [(7, 8, 9, 17), (37, 100, 161)])
def test_rescales_by_blocks_and_by_warps(scale, bins):
    import torch

    wl = _workload(bins, 20, scale)
    P_ref, _, _, st = oracle.solve_batch(wl, oracle.grain_cooling(wl), want_j=False)
    assert st == oracle.OK
    lib = Lib(wl)
    try:
        lib.set_fields(wl.u)
        P, _ = lib.solve(want_j=False, build=heat.HEAT_BUILD_F64)
        r, ok = relerr(P, P_ref)
        assert ok and r <= 1e-10, r
        P1 = torch.empty(wl.n_cells, wl.total_bins, dtype=torch.float64, device="cuda")
        heat.heat_solve_noalloc(lib.ctx, heat.HEAT_BUILD_F64, lib.u, wl.n_cells, P1)
        heat.heat_sync(lib.ctx)
        assert np.array_equal(P, P1.cpu().numpy())
    finally:
        lib.close()
