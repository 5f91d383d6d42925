"""The few-cell recursion where spectra pass the overflow guard: in nearly every run of eight columns, in some of them, and in the
last, partial one, against the FP64 oracle; one warp, four and six warps per spectrum."""
import numpy as np
import pytest

import oracle
from paper_1311_4627_gb300 import heat
from paper_1311_4627_gb300 import workloads as W

from .gpu_helpers import Lib, relerr

pytestmark = pytest.mark.gpu


# fields so strong that X grows by 2^400 to 2^800 in eight states (the guard is at 2^800); the exact path's 1e-10
@pytest.mark.parametrize("scale", [25, 35])
@pytest.mark.parametrize("bins", [(7, 8, 9, 17), (37, 100, 161)])
@pytest.mark.parametrize("cells", [1, 3])
def test_rescales_in_consecutive_runs(scale, bins, cells):
    rng = np.random.default_rng(cells)
    lam = W.wavelength_grid(96)
    u = W.three_bb_fields(lam, 10.0 ** rng.uniform(0, 2, cells), rng.uniform(-1, 1, cells),
                          10.0 ** rng.uniform(-2, 0, (cells, 3))) * 10.0 ** scale
    wl = W.custom(lam, np.geomspace(3.5e-8, 1e-6, len(bins)), ["carbonaceous", "silicate"] * 2, list(bins), u)
    P_ref, _, _, st = oracle.solve_batch(wl, oracle.grain_cooling(wl), want_j=False)
    assert st == oracle.OK
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
