"""The block of the rate matrix that the thermal-discrete back substitution reads: every element it takes lies in the
matrix, and all elements above the diagonal from the column's lowest row on are taken (index arithmetic, on the CPU)."""
from ctypes import c_void_p

import numpy as np
import pytest

from tests.host_build import compile_host

SOURCE = """
#include "gth_tile.cuh"
// marks what the blocks of an nb x nb matrix read; returns the elements read outside it (then not marked)
extern "C" long reads(int nb, const int* low_of, unsigned char* mark) {
    long outside = 0;
    for (int n0 = 0; n0 < nb; n0 += 32)
        for (int lane = 0; lane < 32; ++lane) {
            const int n = n0 + lane, low = n < nb ? low_of[n] : nb;
            for (int i = 0; i < 32; ++i)
                if (heat::gth_tile_in(i, lane, n0, nb, low)) {
                    if (n0 + i < nb && n < nb)
                        mark[(long)(n0 + i) * nb + n] = 1;
                    else
                        ++outside;
                }
        }
    return outside;
}
"""


@pytest.fixture(scope="module")
def host(tmp_path_factory):
    return compile_host(str(tmp_path_factory.mktemp("gth_tile")), SOURCE)


@pytest.mark.parametrize("nb", [2, 3, 31, 32, 33, 63, 64, 65, 97, 100, 128, 150, 161])
def test_reads_stay_in_the_matrix(host, nb):
    rng = np.random.default_rng(nb)
    n = np.arange(nb)
    for low in (np.zeros(nb, np.int32), (n * rng.random(nb)).astype(np.int32), np.maximum(n - 1, 0).astype(np.int32)):
        mark = np.zeros((nb, nb), np.uint8)
        assert host.reads(nb, low.ctypes.data_as(c_void_p),
                          mark.ctypes.data_as(c_void_p)) == 0
        want = (n[:, None] < n) & (n[:, None] >= low) & (n[:, None] // 32 == n // 32)
        assert np.array_equal(mark.astype(bool), want)
