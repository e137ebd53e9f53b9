"""Host side of the decode groups on the 5th-generation tensor cores, without a GPU."""
import ctypes

import pytest

from paper_2602_05269_b200 import build as hgf_build


@pytest.fixture(scope="module")
def lib():
    hgf_build.build()
    from paper_2602_05269_b200 import hgf
    return hgf.lib()


@pytest.mark.parametrize("sets,bytes_a_tile,cols", [(1, 320, 320), (2, 320, 320), (2, 256, 256)], ids=["base3-m8", "base3-m16", "two-bit-m16"])
def test_ring_has_six_stages_wherever_they_fit(lib, sets, bytes_a_tile, cols):
    """Activations of every row length: the ring and the activations' region stay inside the shared memory, the region holds the
    largest problem, and six stages are kept wherever they fit beside it."""
    out = (ctypes.c_int32 * 4)()
    for K in range(64, 16384, 64):
        image = 8 * sets * bytes_a_tile * -(-K // cols)
        fits = lib.hgf_internal_decode_tc_layout(image, out)
        x, stages, stage, room = out
        whole = -(-image // 1024) * 1024
        assert bool(fits) == (whole + 4 * stage <= room), K
        if fits:
            assert x % 1024 == 0 and whole <= x <= 2 * whole and x + stages * stage <= room, (K, x, stages)
            assert stages % 2 == 0 and 4 <= stages <= 10
            assert stages >= 6 or whole + 6 * stage > room, (K, x, stages)
