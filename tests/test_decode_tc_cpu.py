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


def takes(lib, layers, M, r=32, base3=False, sms=148):
    from paper_2602_05269_b200 import hgf
    K, N = ((ctypes.c_int32 * len(layers))(*v) for v in zip(*layers))
    most = ctypes.c_int32()
    return bool(lib.hgf_internal_group_on_tensor_memory(K, N, len(layers), r, M, hgf.FLAG_BASE3 if base3 else 0, sms, ctypes.byref(most)))


def block(d, ffn):
    return [(d, d)] * 4 + [(d, ffn)] * 2 + [(ffn, d)]


# One B200 (148 SMs): the warp MMA's time over the tensor-memory kernel's, whole group in a captured chain
@pytest.mark.parametrize("layers,M,r,base3,ratio", [
    (block(2048, 5632) * 36, 16, 32, False, 1.08), (block(4096, 11008) * 8, 1, 64, True, 1.16), (block(2048, 5632), 9, 32, False, 1.17),
    (block(512, 1408), 16, 32, False, 1.48), (block(1024, 2816), 8, 32, True, 1.08), ([(4096, 11008)] * 2, 1, 64, True, 1.18),
    ([(2048, 5632)] * 2, 16, 32, False, 1.07), ([(4096, 4096)] * 3, 16, 64, False, 1.16), ([(3200, 3200)], 1, 64, True, 1.20),
    ([(768, 208), (3200, 312)], 9, 16, False, 1.49), ([(1024, 256)], 1, 16, True, 1.16), ([(1024, 2048)], 1, 64, True, 0.94),
    ([(5632, 2048)], 1, 32, True, 0.82), ([(5632, 2048)], 16, 32, False, 0.86), ([(11008, 4096)], 8, 64, True, 0.86),
    ([(2048, 2048)], 1, 32, True, 0.91), ([(4096, 4096)], 16, 64, False, 0.95), ([(8192, 1536)], 1, 32, True, 0.73),
    ([(5632, 2048)] * 3, 16, 32, False, 0.90), ([(2048, 2056), (320, 136), (5632, 520), (256, 128)], 16, 32, False, 0.91),
])
def test_groups_go_to_the_faster_kernel(lib, layers, M, r, base3, ratio):
    assert takes(lib, layers, M, r, base3) == (ratio > 1)


def test_groups_that_the_tensor_memory_kernel_cannot_take(lib):
    assert not takes(lib, block(2048, 5632), 8)                     # two-bit weights, up to eight tokens
    assert not takes(lib, block(2048, 8704) * 8, 16)                # activations that leave no room for the ring
    assert not takes(lib, [(64, 16)] * (148 * 33), 16)              # more runs of row tiles on a CTA than its table holds
    assert takes(lib, [(64, 16)] * (148 * 31), 16)
    assert not takes(lib, block(512, 1408), 16, sms=0)              # no device
