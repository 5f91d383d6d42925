"""The thermal-discrete state reduction (panels of states, one block or a cluster per spectrum) against the FP64 oracle
on the same downward rates: bin counts around multiples of the panel, dense matrices, matrices with runs of states that
only step down by one, and both block counts per spectrum (few spectra share each between blocks)."""
import numpy as np
import pytest

import oracle
from paper_1311_4627_gb300 import heat
from paper_1311_4627_gb300 import workloads as W

from .gpu_helpers import Lib, relerr

pytestmark = pytest.mark.gpu


# 1 cell: up to 8 blocks per spectrum; 20 cells x 8 grains: one.  `top`: the highest level in photon energies of the
# shortest wavelength (below 1 every level reaches every other, far above it the upper ones only their neighbours).
# A sum of non-negative products per element: relative error of a few nb ulp, 1e-12 at 300 bins; the bound leaves the
# heating rates' 1e-13 times the length of the chain.
@pytest.mark.parametrize("cells", [1, 20])
@pytest.mark.parametrize("top", [0.5, 3e4])
@pytest.mark.parametrize("bins", [(2, 3, 8, 9, 10, 16, 17, 18), (31, 33, 40, 41, 64, 65, 72, 97), (128, 129, 150, 300)])
def test_panels_and_runs_match_the_oracle(cells, top, bins):
    rng = np.random.default_rng(sum(bins) + cells)
    lam = W.wavelength_grid(64)
    cabs = np.stack([1e-13 * (1 + g) * (1e-5 / lam) ** 1.2 for g in range(len(bins))])
    E = [W.H_PLANCK * W.C_LIGHT / lam[0] * np.geomspace(2e-4, top, nb) * (1 + 0.01 * g) for g, nb in enumerate(bins)]
    T = [np.geomspace(6.0, 3000.0, nb) for nb in bins]
    u = W.three_bb_fields(lam, 10.0 ** rng.uniform(0, 4, cells), rng.uniform(-1, 1, cells),
                          10.0 ** rng.uniform(-2, 0, (cells, 3)))
    off = np.concatenate([[0], np.cumsum(bins)]).astype(np.int32)
    wl = W.Workload("state reduction", lam, np.full(len(bins), 3e-7), ["carbonaceous"] * len(bins), cabs, off,
                    np.concatenate(T), np.concatenate(E), np.ones(len(bins)), u=u)
    lib = Lib(wl)
    try:
        lib.set_fields(wl.u)
        P, _ = lib.solve(want_j=False, build=heat.HEAT_BUILD_F64, cooling=heat.HEAT_COOLING_DISCRETE)
        Dg = heat.heat_get_cooling_discrete(lib.ctx, list(bins))
        P_ref, _, _, st = oracle.solve_batch_discrete(wl, Dg, want_j=False)
        assert st == oracle.OK
        r, ok = relerr(P, P_ref, floor=1e-200)
        assert ok or np.all(P[P_ref <= 1e-200] <= 1.01e-200)
        assert r <= 1e-10, r
    finally:
        lib.close()
