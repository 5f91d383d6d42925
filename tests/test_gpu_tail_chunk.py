"""Exact solves whose last chunk has at most 16 cells: the same bits as in one chunk (the few-cell kernels are chosen by
the cells of the whole solve)."""
import numpy as np
import pytest

from paper_1311_4627_gb300 import heat
from paper_1311_4627_gb300 import workloads as W

from .gpu_helpers import Lib

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tail", [1, 5, 16, 17])
@pytest.mark.parametrize("size_integrate,sign", [(0, 1.0), (1, 1.0), (1, -1.0)])
@pytest.mark.parametrize("point", [False, True])
def test_small_last_chunk(tail, size_integrate, sign, point):
    wl = W.grain_subset(W.batched(cells=32 + tail, n_lambda=96), [0, 30])
    wl.size_weight = np.array([0.75, sign * 0.25])
    lib = Lib(wl)
    try:
        lib.set_fields(wl.u)
        kw = dict(build=heat.HEAT_BUILD_F64, emis=heat.HEAT_EMIS_F64, j_dtype=heat.HEAT_F64,
                  size_integrate=size_integrate, streams=1,
                  heating=heat.HEAT_HEATING_POINT if point else heat.HEAT_HEATING_INTEGRAL)
        P, j = lib.solve(chunk_cells=64, **kw)
        P2, j2 = lib.solve(chunk_cells=32, **kw)
        assert np.array_equal(P, P2) and np.array_equal(j, j2)
    finally:
        lib.close()
