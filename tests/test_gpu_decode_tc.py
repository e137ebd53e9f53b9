"""Groups whose contraction runs on the 5th-generation tensor cores (base-3 weights, or more than eight tokens) against the
oracle: integer results bit for bit, y within the decode path's tolerance."""
import numpy as np
import pytest
import torch

import oracle
from paper_2602_05269_b200 import inputs as syn

TOL = 2e-5   # fp32 accumulation, H kept to ~2^-22: the decode path's


@pytest.fixture(scope="module")
def hgf():
    from paper_2602_05269_b200 import hgf as m
    m.lib()
    return m


def dev(a, dtype=None):
    t = torch.from_numpy(np.ascontiguousarray(a))
    return (t.view(dtype) if dtype is not None else t).cuda()


# (K, N, r, M, gate_group): row tiles that end inside a block of eight and inside a row tile, one column tile, odd and even numbers of
# them in both layouts (K = 320 and 256 are one tile), tokens that fill neither set of eight, no correction, every rank
MIXED = [[(64, 8, 16, 16, 1), (2048, 2056, 32, 16, 1), (320, 136, 0, 9, 1), (5632, 520, 48, 11, 16), (256, 128, 64, 1, 10 ** 6)],
         [(1024, 1000, 64, 12, 1), (704, 72, 32, 16, 64)],
         [(576, 130, 16, 3 + i % 14, 1) for i in range(60)],
         [(5632, 2048, 32, 16, 1)]]


@pytest.mark.gpu
@pytest.mark.parametrize("base3", [False, True])
@pytest.mark.parametrize("shapes", MIXED, ids=["mixed", "two", "many", "long"])
@pytest.mark.parametrize("cap", [16, 8])
def test_group_against_oracle(hgf, shapes, base3, cap):
    if cap == 8 and not base3:
        pytest.skip("two-bit groups of up to eight tokens run elsewhere")
    probs, hosts = [], []
    for i, (K, N, r, M, gg) in enumerate(shapes):
        M = min(M, cap)
        W = syn.make_weights(N, K, config=31, layer=i % 5)
        packed, gamma = hgf.pack_ternary(dev(W), base3=base3)
        T = oracle.ternarise(W, np.float32(gamma))
        x = syn.make_x(M, K, config=31, layer=i)
        q = {"x": dev(x, torch.bfloat16), "packed": packed, "gamma": float(gamma), "d_in": K, "d_out": N,
             "y": torch.zeros((M, N), dtype=torch.float32, device="cuda")}
        h = [x, T, np.float32(gamma), None, None, None]
        if r:
            At, Bt, gate = syn.make_lora(K, N, r, config=31, layer=i)
            gate = gate[:-(-N // gg)]
            q.update(At=dev(At, torch.float16), Bt=dev(Bt, torch.float16), gate=dev(gate), gate_group=gg)
            h[3:] = [At, Bt, np.repeat(gate, min(gg, N))[:N]]
        probs.append(q)
        hosts.append(h)
    group = hgf.Group(probs, flags=hgf.FLAG_BASE3 if base3 else 0)
    y_ints = [torch.full(q["y"].shape, -1, dtype=torch.int32, device="cuda") for q in probs]
    for i, yi in enumerate(y_ints):
        group.debug(i, yi)
    for _ in range(2):  # a second pass over the same buffers gives the same
        group.forward()
    hgf.check_status()
    for i, (q, h, yi) in enumerate(zip(probs, hosts, y_ints)):
        ref = oracle.forward(*h)
        assert np.array_equal(yi.cpu().numpy(), ref["y_int"]), (i, shapes[i])
        err = np.abs(q["y"].cpu().numpy().astype(np.float64) - ref["y"]).max() / np.abs(ref["y"]).max()
        assert err <= TOL, (i, shapes[i], err)
    group.close()


def test_base3_quotients_are_exact_for_every_byte():
    """The operand registers of the base-3 expansion, in the kernel's arithmetic (two bytes in the 16-bit halves of a word).  This is
    the recipe on its own; test_base3_digits_of_every_byte runs the kernel."""
    b = np.arange(256, dtype=np.uint32)
    half = lambda m, c: (b * m + c) >> 8  # noqa: E731  (the byte that the permutation takes)
    assert ((b * 101 + 33) < 65536).all() and ((b * 85 + 85) < 65536).all()
    assert np.array_equal(half(85, 85) & 0xff, b // 3)
    assert np.array_equal(half(57, 0) & 0xfe, 2 * (b // 9))
    assert np.array_equal(half(19, 0) & 0xfe, 2 * (b // 27))
    assert np.array_equal(half(101, 33) & 0x60, 32 * (b // 81))


@pytest.mark.gpu
@pytest.mark.parametrize("M", [3, 16])
def test_base3_digits_of_every_byte(hgf, M):
    """Integer results on packed bytes of all 256 values (242 is the largest a packed matrix holds), against the digits taken apart
    here: one column tile and two, a launch that the tensor cores take."""
    rng = np.random.default_rng(7)
    probs, want = [], []
    for i, K in enumerate((320, 640)):
        steps, N = K // 320, 4096
        raw = rng.integers(0, 256, (N // 16, steps, 16, 64), dtype=np.uint8)
        raw[0, 0, :4] = np.arange(256, dtype=np.uint8).reshape(4, 64)
        q = np.arange(64)
        t, j = q // 16, q % 16
        c = np.empty((N // 16, steps, 16, 320), dtype=np.int64)  # the code of tile column k: a digit of byte q (hgf.h)
        for e in range(5):
            p = j if e < 4 else 16 + j // 4
            k = 32 * (p // 2) + 16 * (p % 2) + 4 * t + (e if e < 4 else j % 4)
            c[..., k] = raw.astype(np.int64) // 3 ** e - (3 * (raw.astype(np.int64) // 3 ** (e + 1)) if e < 4 else 0)
        W = c.transpose(0, 2, 1, 3).reshape(N, K) - 1
        x = syn.make_x(M, K, config=31, layer=70 + i)
        xd = dev(x, torch.bfloat16)
        want.append(hgf.act_quant(xd)[0].cpu().numpy().astype(np.int64) @ W.T)
        packed = dev(raw.reshape(-1))
        for _ in range(6):
            probs.append({"x": xd, "packed": packed, "gamma": 0.5, "d_in": K, "d_out": N,
                          "y": torch.zeros((M, N), dtype=torch.float32, device="cuda")})
    group = hgf.Group(probs, flags=hgf.FLAG_BASE3)
    y_ints = [torch.full(q["y"].shape, -1, dtype=torch.int32, device="cuda") for q in probs]
    for i, yi in enumerate(y_ints):
        group.debug(i, yi)
    group.forward()
    hgf.check_status()
    for i, yi in enumerate(y_ints):
        assert np.array_equal(yi.cpu().numpy(), want[i // 6])
    group.close()
