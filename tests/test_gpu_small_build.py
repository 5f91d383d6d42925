"""The few-cell matrix build (a block per spectrum) against the many-cell build of the same cells, on grids shorter and
longer than a block, of few and many segments per matrix row, with dark segments and a dark cell."""
import numpy as np
import pytest

from paper_1311_4627_gb300 import heat
from paper_1311_4627_gb300 import workloads as W
from tests.gpu_helpers import Lib

pytestmark = pytest.mark.gpu


# FP64: sums of N positive terms in another order, N 2^-53 < 2e-13 on every matrix element; FP32: photon prefixes carry
# N 2^-24 at worst and sqrt(N) 2^-24 typically, 2e-6 at N = 1100; the recursion passes a few of either on to P.
@pytest.mark.parametrize("build,tol", [(heat.HEAT_BUILD_F32, 2e-4), (heat.HEAT_BUILD_F64, 1e-10)])
@pytest.mark.parametrize("cells,n_lambda", [(1, 2), (2, 3), (1, 40), (3, 257), (2, 1100)])
def test_few_cells_equal_many(build, tol, cells, n_lambda):
    lam = W.wavelength_grid(n_lambda)
    rng = np.random.Generator(np.random.PCG64(n_lambda))
    u = W.three_bb_fields(lam, 10.0 ** rng.uniform(-2, 4, 600), rng.uniform(-1, 1, 600),
                          10.0 ** rng.uniform(-2, 0, (600, 3)))
    u[0, : n_lambda // 3] = 0.0
    if cells > 2:
        u[cells - 1] = 0.0
    wl = W.custom(lam, np.array([4e-8, 1e-6, 3e-5]), ["carbonaceous", "silicate", "carbonaceous"], [33, 96, 161], u)
    lib = Lib(wl)
    try:
        lib.set_fields(wl.u)
        P, _ = lib.solve(want_j=False, build=build)
        lib.set_fields(wl.u[:cells])
        Q, _ = lib.solve(want_j=False, build=build)
        floor = 1e-280 if build == heat.HEAT_BUILD_F64 else 1e-20
        big = P[:cells] > floor
        assert np.all(np.abs(Q[big] - P[:cells][big]) <= tol * P[:cells][big])
        assert np.all(Q[~big] <= 2 * floor)
    finally:
        lib.close()
