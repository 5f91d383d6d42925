"""heat_autotune leaves the build's prefetch at its default where the solve's build has none to choose (two passes)."""
import pytest

from paper_1311_4627_gb300 import heat
from paper_1311_4627_gb300 import workloads as W

from .gpu_helpers import Lib

pytestmark = pytest.mark.gpu


def test_no_choice_between_equal_builds():
    import torch

    wl = W.grain_subset(W.batched(cells=150, n_lambda=96), [0, 17, 41])
    lib = Lib(wl)
    try:
        lib.set_fields(wl.u)
        j = torch.empty(wl.n_cells, wl.n_grains, wl.n_lambda, dtype=torch.float32, device="cuda")
        for _ in range(6):
            heat.heat_autotune(lib.ctx, heat.heat_default_opts(build=heat.HEAT_BUILD_F32, emis=heat.HEAT_EMIS_BF16X3,
                                                               j_dtype=heat.HEAT_F32, fused_build=2), None, j,
                               torch.cuda.current_stream().cuda_stream)
            assert heat.heat_get_tuning(lib.ctx)["build_prefetch"] == 0
    finally:
        lib.close()
