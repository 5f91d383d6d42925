"""Pruned recursions of large launches, where no grain's tasks take a block (a kernel without that form), against the same
cells in launches that give the wide grains' tasks a block each: the same bits."""
import numpy as np
import pytest

from paper_1311_4627_gb300 import heat
from paper_1311_4627_gb300 import workloads as W

from .gpu_helpers import Lib

pytestmark = pytest.mark.gpu


# 32 equal grains of 34 bins: a warp alone would be busy for more than a third of the launch below about 10,000 cells
@pytest.mark.parametrize("build", [heat.HEAT_BUILD_F32, heat.HEAT_BUILD_F64])
def test_large_and_small_launches(build):
    rng = np.random.default_rng(11)
    cells, lam = 12001, W.wavelength_grid(48)
    u = W.three_bb_fields(lam, 10.0 ** rng.uniform(-2, 4, cells), rng.uniform(-1, 1, cells),
                          10.0 ** rng.uniform(-2, 0, (cells, 3)))
    wl = W.custom(lam, np.full(32, 4e-7), ["carbonaceous", "silicate"] * 16, [34] * 32, u)
    lib = Lib(wl)
    try:
        lib.set_fields(wl.u)
        P, _ = lib.solve(want_j=False, build=build, prune_eps=1e-9)
        Q, _ = lib.solve(want_j=False, build=build, prune_eps=1e-9, chunk_cells=512, streams=2)
        assert np.array_equal(P, Q)
        assert np.allclose(P[:, :34].sum(axis=1), 1.0)
    finally:
        lib.close()
