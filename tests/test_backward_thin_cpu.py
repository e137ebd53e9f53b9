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


GRADIENTS = ("dx", "dW", "dAt", "dBt", "dgate")


def trace(lib, M, K, N, r, want=GRADIENTS, gamma=0.02, sms=148, pairs=74):
    """A backward pass of which nothing is enqueued: its room for partial sums, what its launches do with it, who rides with dW and with dX."""
    uses, rides, floats = (ctypes.c_int64 * 300)(), (ctypes.c_int32 * 8)(), ctypes.c_int64()
    bits = sum(1 << GRADIENTS.index(n) for n in want)
    n = lib.hgf_internal_backward_trace(ctypes.c_int64(M), ctypes.c_int64(K), ctypes.c_int64(N), r, ctypes.c_float(gamma), bits, sms, pairs, ctypes.byref(floats), uses, 100, rides)
    assert 0 <= n < 100
    return floats.value, [tuple(uses[3 * i:3 * i + 3]) for i in range(n)], list(rides)


SIZES = [(4096, 2112, 2048), (3300, 2048, 2048), (2656, 3456, 3456), (2500, 2112, 512), (4096, 2176, 3072), (3456, 3968, 3200), (3072, 3072, 3072), (4096, 2560, 2560),
         (2560, 2560, 2560), (2261, 1024, 2048), (8192, 2048, 5632), (64, 512, 512), (1, 64, 8)]
WANTS = [GRADIENTS, ("dW", "dAt", "dBt", "dgate"), ("dW", "dAt", "dgate"), ("dx", "dAt", "dBt"), ("dW", "dBt"), ("dgate",)]


@pytest.mark.parametrize("gamma", [0.02, 0.0])
@pytest.mark.parametrize("want", WANTS, ids="-".join)
@pytest.mark.parametrize("sms", [148, 132, 20])
def test_partial_sums_are_read_before_their_room_is_written_again(lib, sms, want, gamma):
    rng = random.Random(sms)
    sizes = SIZES + [(rng.randint(1, 9000), 64 * rng.randint(1, 130), 8 * rng.randint(1, 1000)) for _ in range(60)]
    sizes += [(256 * m, 256 * k, 256 * n) for m in (4, 8, 10, 16) for k in (4, 8, 10, 16) for n in (2, 8, 12)]
    for M, K, N in sizes:
        floats, uses, rides = trace(lib, M, K, N, rng.choice([16, 32, 48, 64]), want, gamma, sms, sms // 2)
        unread = {}  # first float -> end, of the sums that are still to be read
        for write, first, end in uses:
            assert 0 <= first < end <= floats
            if write:
                assert all(end <= a or first >= b for a, b in unread.items()), f"{M} x {K} -> {N}, {rides}: sums written over others that are still to be read"
                unread[first] = end
            else:
                assert unread.pop(first, None) == end, f"{M} x {K} -> {N}, {rides}: other sums are read than were written"
        assert not unread
