"""Heating rates of the thermal-discrete solve on grids where a window lies inside one segment, spans a few or all of
them, meets dark segments or slopes too steep for the fixed-point integral (|slope x log width| >= 1), with row
lengths around the warp's 32 bins: P and j against the FP64 oracle on the same downward rates."""
import numpy as np
import pytest

import oracle
from paper_1311_4627_gb300 import heat
from paper_1311_4627_gb300 import workloads as W

from .gpu_helpers import Lib, relerr

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_lambda,nb", [(2, 2), (2, 33), (3, 65), (9, 32), (40, 31), (300, 64)])
def test_discrete_rates_on_coarse_and_uneven_grids(n_lambda, nb):
    rng = np.random.default_rng(100 * n_lambda + nb)
    lam = np.exp(np.linspace(np.log(1e-5), np.log(1e-1), n_lambda))
    lam[1:-1] *= np.exp(rng.uniform(-0.3, 0.3, n_lambda - 2) * np.log(lam[1] / lam[0]))
    cabs = 1e-13 * (1e-5 / lam) ** 1.3
    E = W.H_PLANCK * W.C_LIGHT * np.geomspace(20.0, 2e5, nb)  # photons of 0.05 um .. 500 um
    u = 1e-14 * np.exp(rng.normal(0.0, 1.5, (3, n_lambda)))
    if n_lambda > 8:
        u[1, n_lambda // 2] = 0.0  # two dark segments
    wl = W.Workload("coarse grid", lam, np.array([3e-7]), ["carbonaceous"], cabs[None, :],
                    np.array([0, nb], dtype=np.int32), np.geomspace(4.0, 2500.0, nb), E, np.ones(1), u=u)
    lib = Lib(wl)
    try:
        lib.set_fields(wl.u)
        opts = dict(build=heat.HEAT_BUILD_F64, emis=heat.HEAT_EMIS_F64, j_dtype=heat.HEAT_F64,
                    cooling=heat.HEAT_COOLING_DISCRETE)
        P, j = lib.solve(**opts)
        Dg = heat.heat_get_cooling_discrete(lib.ctx, [nb])
        P_ref, j_ref, _, st = oracle.solve_batch_discrete(wl, Dg, want_ledger=True)
        assert st == oracle.OK
        # a rate is off by a few ulp of its segment's integral over a window of >= 1/100 of the segment (1e-13), the
        # state reduction multiplies up to nb of them
        for got, ref in ((P, P_ref), (j, j_ref)):
            r, ok = relerr(got, ref)
            assert ok and r <= 1e-10, r
    finally:
        lib.close()
