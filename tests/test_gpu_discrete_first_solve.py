"""The first thermal-discrete solve of a grain set, which makes the rate tables and the launch order, on a non-blocking
stream and over two internal streams: the bits of the later solves."""
import numpy as np
import pytest

from paper_1311_4627_gb300 import heat
from paper_1311_4627_gb300 import workloads as W

from .gpu_helpers import Lib

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("streams", [1, 2])
def test_first_solve_on_a_non_blocking_stream(streams):
    import torch

    wl = W.grain_subset(W.batched(cells=70, n_lambda=96), [0, 30, 1])
    lib = Lib(wl)
    try:
        lib.set_fields(wl.u)
        torch.cuda.synchronize()
        s = torch.cuda.Stream()
        o = heat.heat_default_opts(build=heat.HEAT_BUILD_F64, cooling=heat.HEAT_COOLING_DISCRETE, streams=streams,
                                   chunk_cells=32, emis=heat.HEAT_EMIS_NONE)
        out = []
        for _ in range(3):
            P = torch.zeros(wl.n_cells, wl.total_bins, dtype=torch.float64, device="cuda")
            torch.cuda.synchronize()
            heat.heat_solve(lib.ctx, o, P, None, s.cuda_stream)
            heat.heat_sync(lib.ctx)
            out.append(P.cpu().numpy())
        assert np.all(out[0].sum(axis=1) > 2.9)
        assert np.array_equal(out[0], out[1]) and np.array_equal(out[0], out[2])
    finally:
        lib.close()
