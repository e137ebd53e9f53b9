"""How the thin products of the backward pass are dealt to the pairs of CTAs (tc_deal_thin), without a GPU."""
import ctypes
import random

import pytest

from paper_2602_05269_b200 import build as hgf_build


@pytest.fixture(scope="module")
def lib():
    hgf_build.build()
    from paper_2602_05269_b200 import hgf
    return hgf.lib()


def deal(lib, products, num_work, n_half, kb_all, pairs):
    I, Cn = ((ctypes.c_int32 * len(products))(*v) for v in zip(*products))
    out = (ctypes.c_int32 * 9)()
    ride = lib.hgf_internal_tc_deal_thin(I, Cn, len(products), num_work, n_half, kb_all, pairs, out)
    return bool(ride), list(out)


@pytest.mark.parametrize("pairs", [74, 73, 7, 1])
def test_every_part_of_every_tile_goes_to_one_pair(lib, pairs):
    rng = random.Random(pairs)
    sizes = [(8, 64), (256, 64), (257, 8192), (5632, 8192), (8192, 5632), (2048, 450)] + [(rng.randint(1, 9000), rng.randint(1, 9000)) for _ in range(60)]
    rode = 0
    for k, first in enumerate(sizes):
        for products in ([first], [first, sizes[(7 * k + 3) % len(sizes)]]):
            num_work = rng.choice([1, pairs, 2 * pairs, rng.randint(1, 4 * pairs)])
            n_half = 2 * (rng.randint(0, pairs // 2)) if num_work > pairs else 0
            ride, (items, items0, busy, c_idle, c_busy, *parts) = deal(lib, products, num_work, n_half, rng.randint(7, 200), pairs)
            if not ride:  # (launches of their own)
                assert items == c_idle == c_busy == 0
                continue
            rode += 1
            # the pieces in the order in which the kernel numbers them: (product, tile, part), none of them without a block
            pieces = []
            for i, (I, Cn) in enumerate(products):
                blocks, splits, per = -(-Cn // 64), parts[2 * i], parts[2 * i + 1]
                assert 1 <= splits <= 4 and (splits - 1) * per < blocks <= splits * per
                pieces += [(i, tile, part) for part in range(splits) for tile in range(-(-I // 256))]
            assert items == len(pieces) and items0 == sum(p[0] == 0 for p in pieces) and busy == num_work % pairs
            taken = []
            for pair in range(pairs):
                first_piece, many = ((pairs - busy) * c_idle + pair * c_busy, c_busy) if pair < busy else ((pair - busy) * c_idle, c_idle)
                taken += range(first_piece, min(items, first_piece + many))
            assert sorted(taken) == list(range(items))
    assert rode > 5 or pairs == 1


# (M, K, N, whether dH and G ride behind dW, whether dA rides behind dX): training steps that take less time so
@pytest.mark.parametrize("M,K,N,dw,dx", [(2048, 2048, 2048, True, True), (700, 1024, 3000, True, True), (8000, 768, 1536, True, True), (8192, 4096, 1024, True, True),
                                         (8192, 2048, 5632, True, False)])
def test_where_they_ride(lib, M, K, N, dw, dx):
    def product(I, J, blocks, thin):
        tiles = -(-I // 256) * -(-J // 256)
        half = 2 * (tiles % 74) if tiles > 74 and 2 * (tiles % 74) <= 74 and J % 256 == 0 else 0
        return deal(lib, thin, tiles + half // 2, half, blocks, 74)[0]
    assert product(N, K, -(-M // 64), [(M, N), (N, M)]) == dw
    assert product(M, K, -(-N // 64) + 1, [(K, M)]) == dx
