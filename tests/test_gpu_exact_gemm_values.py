"""The exact emissivity's fixed-point contraction on values outside the ordinary: zeros of either sign, subnormals, infinities."""
import numpy as np
import pytest

from paper_1311_4627_gb300 import heat
from paper_1311_4627_gb300 import workloads as W

from .gpu_helpers import Lib

pytestmark = pytest.mark.gpu

EXACT = dict(build=heat.HEAT_BUILD_F64, emis=heat.HEAT_EMIS_F64, j_dtype=heat.HEAT_F64)


def _workload(cells, n_lambda=64):
    return W.grain_subset(W.batched(cells=cells, n_lambda=n_lambda), [0, 30])


def test_negative_zeros():
    """Cross-sections and size weights of -0 count as 0: the same j."""
    wl = _workload(33)
    wl.cabs = wl.cabs.copy()
    wl.cabs[:, ::5] = 0.0
    wl.size_weight = np.array([0.0, 0.5])
    out = []
    for sign in (1.0, -1.0):
        wl.cabs[:, ::5] = sign * 0.0
        wl.size_weight[0] = sign * 0.0
        lib = Lib(wl)
        try:
            lib.set_fields(wl.u)
            out.append((lib.solve(**EXACT)[1], lib.solve(size_integrate=1, **EXACT)[1]))
        finally:
            lib.close()
    assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1])
    assert np.all(out[0][1] >= 0.0) and out[0][1].max() > 0.0


def test_subnormal_emissivities():
    """Emission far below the normal range (size weights of 1e-300): j as the few-cell kernel's FMA sums give it, to the
    exact path's 1e-10 and a few units in the last place of a subnormal."""
    wl = _workload(33)
    wl.size_weight = np.array([1e-300, 1e-302])
    lib = Lib(wl)
    try:
        lib.set_fields(wl.u)
        _, j = lib.solve(size_integrate=1, **EXACT)
        lib.set_fields(wl.u[:3])
        _, few = lib.solve(size_integrate=1, **EXACT)
    finally:
        lib.close()
    assert np.any((few > 0.0) & (few < 2.0**-1022))
    assert np.all(np.abs(j[:3] - few) <= 1e-10 * few + 8 * 2.0**-1074)


def test_infinite_kernels():
    """Size weights that take part of the emission kernel, or only sums of it, beyond the range: infinities, NaN and finite j
    where the few-cell kernel's FMA sums have them."""
    wl = _workload(33)
    wl.cabs = wl.cabs * 1e10
    wl.size_weight = np.array([1e307, 1e308])
    lib = Lib(wl)
    try:
        lib.set_fields(wl.u)
        _, j = lib.solve(size_integrate=1, **EXACT)
        lib.set_fields(wl.u[:3])
        _, few = lib.solve(size_integrate=1, **EXACT)
    finally:
        lib.close()
    assert np.any(~np.isfinite(few)) and np.any(np.isfinite(few))
    assert np.array_equal(np.isnan(j[:3]), np.isnan(few)) and np.array_equal(np.isinf(j[:3]), np.isinf(few))
    ok = np.isfinite(few)
    assert np.all(np.abs(j[:3][ok] - few[ok]) <= 1e-10 * few[ok])
