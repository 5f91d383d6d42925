"""The thermal-discrete solve on a rate-matrix buffer that an earlier, larger solve filled with rates that overflow: bin
counts that are no multiple of the back substitution's 32 columns, so that its last block ends past the matrix."""
import numpy as np
import pytest

import oracle
from paper_1311_4627_gb300 import heat
from paper_1311_4627_gb300 import workloads as W

from .gpu_helpers import Lib, relerr

pytestmark = pytest.mark.gpu

DISCRETE = dict(build=heat.HEAT_BUILD_F64, cooling=heat.HEAT_COOLING_DISCRETE)


def _workload(bins, cells, scale=1.0):
    rng = np.random.default_rng(sum(bins))
    lam = W.wavelength_grid(64)
    cabs = np.stack([1e-13 * (1 + g) * (1e-5 / lam) ** 1.2 for g in range(len(bins))])
    E = [W.H_PLANCK * W.C_LIGHT / lam[0] * np.geomspace(2e-4, 0.5, nb) * (1 + 0.01 * g) for g, nb in enumerate(bins)]
    T = [np.geomspace(6.0, 3000.0, nb) for nb in bins]
    u = scale * W.three_bb_fields(lam, 10.0 ** rng.uniform(0, 4, cells), rng.uniform(-1, 1, cells),
                                  10.0 ** rng.uniform(-2, 0, (cells, 3)))
    off = np.concatenate([[0], np.cumsum(bins)]).astype(np.int32)
    return W.Workload("buffer reuse", lam, np.full(len(bins), 3e-7), ["carbonaceous"] * len(bins), cabs, off,
                      np.concatenate(T), np.concatenate(E), np.ones(len(bins)), u=u)


# 1e-10 as every thermal-discrete comparison with the oracle
@pytest.mark.parametrize("bins", [(33,), (100,), (63, 65, 97), (129, 150)])
def test_what_an_earlier_solve_left_does_not_count(bins):
    big = _workload((160, 160, 160), 6, scale=1e300)  # rates up to infinity
    lib = Lib(big)
    try:
        lib.set_fields(big.u)
        try:
            lib.solve(want_j=False, **DISCRETE)
        except heat.HeatError:
            pass  # overflowing rates may be reported
        wl = _workload(bins, 3)
        heat.heat_set_grains(lib.ctx, wl.radius, wl.cabs, wl.bin_off, wl.T, wl.E, wl.size_weight)
        lib.wl = wl
        lib.set_fields(wl.u)
        P, _ = lib.solve(want_j=False, **DISCRETE)
        Dg = heat.heat_get_cooling_discrete(lib.ctx, list(bins))
        P_ref, _, _, st = oracle.solve_batch_discrete(wl, Dg, want_j=False)
        assert st == oracle.OK
        r, _ = relerr(P, P_ref, floor=1e-200)
        assert r <= 1e-10, r
    finally:
        lib.close()
