"""The exact emissivity's fixed-point contraction at the edges of its tiles (64 cells x 32 wavelengths,
bins four and sixteen at a time) against the FP64 oracle, and the FP64 form that kernels with a negative
size weight take.  Tolerance: the exact path's 1e-10 on every entry above 1e-280."""
import numpy as np
import pytest

import oracle
from paper_1311_4627_gb300 import heat
from paper_1311_4627_gb300 import workloads as W
from tests.gpu_helpers import Lib, relerr

pytestmark = pytest.mark.gpu


def workload(cells, n_lambda, bins, seed=5):
    lam = W.wavelength_grid(n_lambda)
    G = len(bins)
    rng = np.random.Generator(np.random.PCG64(seed))
    u = W.three_bb_fields(lam, 10.0 ** rng.uniform(-2, 4, cells), rng.uniform(-1, 1, cells),
                          10.0 ** rng.uniform(-2, 0, (cells, 3)))
    return W.custom(lam, np.geomspace(4e-8, 2e-5, G), ["carbonaceous", "silicate"][:1] * G, bins, u)


@pytest.mark.parametrize("cells,n_lambda,bins", [(17, 31, [2, 5]), (64, 33, [16, 17]), (65, 32, [70]),
                                                 (130, 65, [3, 33, 48])])
def test_exact_emissivity_at_tile_edges(cells, n_lambda, bins):
    wl = workload(cells, n_lambda, bins)
    _, j_ref, _, st = oracle.solve_batch(wl, oracle.grain_cooling(wl))
    assert st == oracle.OK
    lib = Lib(wl)
    try:
        lib.set_fields(wl.u)
        _, j = lib.solve()
    finally:
        lib.close()
    r, ok = relerr(j, j_ref)
    assert ok and r <= 1e-10, r


@pytest.mark.parametrize("sign", [1.0, -1.0])
def test_size_integrated_weights_of_either_sign(sign):
    wl = workload(33, 40, [17, 24])
    wl.size_weight = np.array([0.75, sign * 0.25])
    _, j_ref, _, st = oracle.solve_batch(wl, oracle.grain_cooling(wl))
    assert st == oracle.OK
    ref = 0.75 * j_ref[:, 0] + sign * 0.25 * j_ref[:, 1]
    lib = Lib(wl)
    try:
        lib.set_fields(wl.u)
        _, j = lib.solve(size_integrate=1)
    finally:
        lib.close()
    scale = 0.75 * j_ref[:, 0] + 0.25 * j_ref[:, 1]
    assert np.all(np.abs(j - ref) <= 1e-10 * scale + 1e-290)
