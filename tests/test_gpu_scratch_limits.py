"""Solves at the limit of the device's memory, the rest of which the test holds: the two-pass build's prefix table is
optional, so a solve that has room for everything else succeeds, in a graph too, with the same bits."""
import numpy as np
import pytest

from paper_1311_4627_gb300 import heat
from paper_1311_4627_gb300 import workloads as W

from .gpu_helpers import Lib

pytestmark = pytest.mark.gpu

# 8 grains of 2 to 4 bins on 2000 wavelengths, 2 chunks of 4096 cells: per chunk field tables of 131 MB, a prefix table of
# 524 MB, everything else below 10 MB
CELLS, CHUNK, FIELDS, PREFIX = 8192, 4096, 131 << 20, 524 << 20
OPTS = dict(build=heat.HEAT_BUILD_F64, emis=heat.HEAT_EMIS_NONE, chunk_cells=CHUNK)


@pytest.fixture(scope="module")
def workload():
    rng = np.random.default_rng(3)
    lam = W.wavelength_grid(2000)
    u = W.three_bb_fields(lam, 10.0 ** rng.uniform(0, 4, CELLS), rng.uniform(-1, 1, CELLS),
                          10.0 ** rng.uniform(-2, 0, (CELLS, 3)))
    return W.custom(lam, np.geomspace(4e-8, 1e-6, 8), ["carbonaceous", "silicate"] * 4, [2, 3, 4, 3] * 2, u)


class _Hold:
    """Device memory taken away until `leave` bytes are free."""

    def __init__(self, leave):
        import torch

        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        free, _ = torch.cuda.mem_get_info()
        self.block = torch.empty(free - leave, dtype=torch.uint8, device="cuda")

    def release(self):
        import torch

        self.block = None
        torch.cuda.empty_cache()


def _solve(lib, P, stream=None, **opts):
    import torch

    P.zero_()
    torch.cuda.synchronize()
    heat.heat_solve(lib.ctx, heat.heat_default_opts(**dict(OPTS, **opts)), P, None,
                    stream or torch.cuda.current_stream().cuda_stream)
    heat.heat_sync(lib.ctx)
    return P.cpu().numpy()


@pytest.fixture()
def lib_and_P(workload):
    import torch

    P = torch.empty(CELLS, workload.total_bins, dtype=torch.float64, device="cuda")
    lib = Lib(workload)
    lib.set_fields(workload.u)
    ref = _solve(lib, P, streams=2)
    lib.close()
    lib = Lib(workload)
    lib.set_fields(workload.u)
    yield lib, P, ref
    lib.close()


def test_no_room_for_the_prefix_table(lib_and_P):
    """Room for both chunks' scratch, or one chunk's and its prefix table: the scratch comes first."""
    import torch

    lib, P, ref = lib_and_P
    s = torch.cuda.Stream()
    hold = _Hold(FIELDS + PREFIX + (60 << 20))
    try:
        for _ in range(2):
            assert np.array_equal(_solve(lib, P, streams=2), ref)
        g = heat.Graph(lib.ctx, heat.heat_default_opts(streams=2, **OPTS), P, None, s.cuda_stream)
        P.zero_()
        torch.cuda.synchronize()
        g.launch(s.cuda_stream)
        s.synchronize()
        assert np.array_equal(P.cpu().numpy(), ref)
        g.close()
    finally:
        hold.release()
    assert np.array_equal(_solve(lib, P, streams=2), ref)  # with the table again


def test_the_prefix_table_gives_way(lib_and_P):
    """A second stream's scratch where only the first one's prefix table can make room for it."""
    lib, P, ref = lib_and_P
    assert np.array_equal(_solve(lib, P, streams=1), ref)
    hold = _Hold(FIELDS // 2)
    try:
        assert np.array_equal(_solve(lib, P, streams=2), ref)
    finally:
        hold.release()


# 2 GB of chunk scratch (45 % of 4 GB) hold about 2097 groups of 32 cells by their field tables, 419 with a prefix table
@pytest.mark.parametrize("opts,chunks", [(dict(heating=heat.HEAT_HEATING_POINT), 1), ({}, 2)])
def test_only_the_two_pass_build_makes_room_for_its_table(workload, opts, chunks):
    """The default chunk of a solve without a prefix table (the point rule) does not shrink for one; kernel launches of a
    captured solve against those of one chunk of all cells."""
    import torch

    cells = 2 * CELLS
    P = torch.empty(cells, workload.total_bins, dtype=torch.float64, device="cuda")
    lib = Lib(workload)
    s = torch.cuda.Stream()
    hold = None
    try:
        lib.set_fields(np.concatenate([workload.u, workload.u]))
        hold = _Hold(4 << 30)
        nodes = []
        for chunk in (0, cells):
            g = heat.Graph(lib.ctx, heat.heat_default_opts(**dict(OPTS, streams=1, chunk_cells=chunk, **opts)), P, None,
                           s.cuda_stream)
            nodes.append(g.kernel_nodes())
            g.close()
        assert nodes[0] == chunks * nodes[1]
    finally:
        if hold:
            hold.release()
        lib.close()


def test_a_small_table_does_not_shrink_the_chunk():
    """A prefix table of a tenth of the rest (one grain of 180 bins that all reach each other, 2000 wavelengths: 5.2 MB per 32
    cells, 0.5 MB of table): 2 GB hold 412 groups without it, 375 with it; 395 are still one chunk."""
    import torch

    cells, lam = 395 * 32, W.wavelength_grid(2000)
    u = W.three_bb_fields(lam, np.full(cells, 10.0), np.zeros(cells), np.full((cells, 3), 0.3))
    wl = W.custom(lam, np.array([3.5e-8]), ["carbonaceous"], [180], u)
    P = torch.empty(cells, wl.total_bins, dtype=torch.float64, device="cuda")
    lib = Lib(wl)
    s = torch.cuda.Stream()
    hold = None
    try:
        lib.set_fields(wl.u)
        hold = _Hold(4 << 30)
        nodes = []
        for chunk in (0, cells):
            g = heat.Graph(lib.ctx, heat.heat_default_opts(**dict(OPTS, streams=1, chunk_cells=chunk)), P, None, s.cuda_stream)
            nodes.append(g.kernel_nodes())
            g.close()
        assert nodes[0] == nodes[1]
    finally:
        if hold:
            hold.release()
        lib.close()


@pytest.mark.parametrize("prefetch", [1, 2])
def test_one_walk_prefetch_on_and_off(workload, prefetch):
    """The FP32 build without room for its prefix table (half the bytes of FP64), with and without its pattern prefetch."""
    import torch

    P = torch.empty(CELLS, workload.total_bins, dtype=torch.float64, device="cuda")
    lib = Lib(workload)
    hold = None
    try:
        lib.set_fields(workload.u)
        opts = dict(build=heat.HEAT_BUILD_F32, streams=1)
        hold = _Hold((FIELDS + PREFIX) // 2 - (60 << 20))
        a = _solve(lib, P, build_prefetch=prefetch, **opts)
        hold.release()
        assert np.array_equal(a, _solve(lib, P, **opts))
    finally:
        if hold:
            hold.release()
        lib.close()
