"""The few-cell FP32 build cut into 1 to 16 parts per spectrum, against the many-cell build of the same cells: the same
bits, on grids of one segment (all elements in one part), of fewer segments than parts, and of many."""
import numpy as np
import pytest

from paper_1311_4627_gb300 import heat
from paper_1311_4627_gb300 import workloads as W

from .gpu_helpers import Lib

pytestmark = pytest.mark.gpu


# 304 blocks over cells x grains: 16 parts (1 cell x 3 grains), 14 (7 x 3), 7 (13 x 3), 6 (16 x 3), 1 (16 x 19)
@pytest.mark.parametrize("cells,grains", [(1, 3), (7, 3), (13, 3), (16, 3), (16, 19)])
@pytest.mark.parametrize("n_lambda", [2, 3, 9, 40, 601])
def test_parts_give_the_many_cell_bits(cells, grains, n_lambda):
    rng = np.random.default_rng(n_lambda)
    lam = W.wavelength_grid(n_lambda)
    u = W.three_bb_fields(lam, 10.0 ** rng.uniform(-2, 4, 40), rng.uniform(-1, 1, 40), 10.0 ** rng.uniform(-2, 0, (40, 3)))
    u[0, : n_lambda // 3] = 0.0
    wl = W.custom(lam, np.geomspace(3.5e-8, 3e-6, grains), ["carbonaceous"] * grains, [2, 33, 150] + [20] * (grains - 3), u)
    lib = Lib(wl)
    try:
        lib.set_fields(wl.u)
        opts = dict(build=heat.HEAT_BUILD_F32, want_j=False)
        P, _ = lib.solve(**opts)
        Q, _ = lib.solve(cell_count=cells, **opts)
        assert np.array_equal(P[:cells], Q)
    finally:
        lib.close()
