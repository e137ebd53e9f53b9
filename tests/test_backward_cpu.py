"""Host side of the backward pass, without a GPU."""
import pytest

from paper_2602_05269_b200 import build as hgf_build


@pytest.fixture(scope="module")
def lib():
    hgf_build.build()
    from paper_2602_05269_b200 import hgf
    return hgf.lib()


# One B200 (148 SMs, 74 pairs), the product alone: single CTAs' time over pairs'
@pytest.mark.parametrize("I,J,C,pairs", [
    (8192, 2048, 5632, True), (5632, 2048, 8192, True),     # the large products of a training step: 1.16, 1.09
    (512, 512, 8192, True), (136, 192, 2048, True),         # 1.25, 1.16
    (4096, 4096, 300, False), (2048, 12544, 256, False),    # short contractions: 0.91, 0.91
    (136, 192, 64, False), (304, 8192, 64, False),          # 0.96, 0.97
    (304, 12544, 1024, False), (384, 12544, 2048, False),   # 147 tiles of 128 rows are one round, 98 of 256 rows one and a half: 0.96, 0.95
    (304, 8192, 1024, True), (640, 8192, 1024, True),       # as many rounds either way: 1.03, 1.03
    (512, 2048, 448, True), (304, 4096, 448, True),         # one round of tiles: 1.03, 1.05
    (4096, 4096, 448, False), (640, 8192, 512, False),      # several: 0.94, 0.96
    (1152, 8192, 640, False), (2176, 6656, 768, False),     # half a round more: 0.93, 0.98
    (2176, 6656, 2048, True), (1152, 10496, 4096, True),    # the same with a long contraction: 1.16, 1.10
    (128, 4096, 4096, False), (4096, 128, 4096, False),     # outputs that are no larger than one tile of a single CTA
])
def test_products_that_pairs_of_ctas_take(lib, I, J, C, pairs):
    assert bool(lib.hgf_internal_tc_pairs_pay(I, J, C, 148, 74)) == pairs
