"""Groups whose contraction runs on the 5th-generation tensor cores (base-3 weights, or more than eight tokens) against the
oracle: integer results bit for bit, y within the decode path's tolerance."""
import ctypes

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


# Small layers behind the ones of a case: without them the launch would stay on the warp MMA (see decode_tc_pays).
FILL = [(320, 1000, 16, 16, 1)] * 16


def most_problems(hgf, shapes, base3, cap):
    """The largest number of problems in a CTA's share on 148 SMs if the tensor-memory kernel takes the group, else 0."""
    K, N, M = [s[0] for s in shapes], [s[1] for s in shapes], max(min(s[3], cap) for s in shapes)
    most, arr = ctypes.c_int32(), ctypes.c_int32 * len(shapes)
    on = hgf.lib().hgf_internal_group_on_tensor_memory(arr(*K), arr(*N), len(K), 32, M, hgf.FLAG_BASE3 if base3 else 0, 148, ctypes.byref(most))
    return most.value if on else 0


def check_group(hgf, shapes, base3, cap, *, flags=0, bf16=False, variants=5):
    probs, hosts, made = [], [], {}
    for i, (K, N, r, M, gg) in enumerate(shapes):
        M = min(M, cap)
        key = (K, N, i % variants)
        if key not in made:
            W = syn.make_weights(N, K, config=31, layer=i % variants)
            packed, gamma = hgf.pack_ternary(dev(W), base3=base3)
            made[key] = packed, gamma, oracle.ternarise(W, np.float32(gamma))
        packed, gamma, T = made[key]
        x = syn.make_x(M, K, config=31, layer=i)
        q = {"x": dev(x, torch.bfloat16), "packed": packed, "gamma": float(gamma), "d_in": K, "d_out": N,
             "y": torch.zeros((M, N), dtype=torch.bfloat16 if bf16 else torch.float32, device="cuda")}
        h = [x, T, np.float32(gamma), None, None, None]
        if r:
            At, Bt, gate = syn.make_lora(K, N, r, config=31, layer=i)
            gate = gate[:-(-N // gg)]
            q.update(At=dev(At, torch.float16), Bt=dev(Bt, torch.float16), gate=dev(gate), gate_group=gg)
            h[3:] = [At, Bt, np.repeat(gate, min(gg, N))[:N]]
        probs.append(q)
        hosts.append(h)
    group = hgf.Group(probs, flags=flags | (hgf.FLAG_BASE3 if base3 else 0) | (hgf.FLAG_OUT_BF16 if bf16 else 0))
    y_ints = [torch.full(q["y"].shape, -1, dtype=torch.int32, device="cuda") for q in probs]
    for i, yi in enumerate(y_ints):
        group.debug(i, yi)
    for _ in range(2):  # a second pass over the same buffers gives the same
        group.forward()
    hgf.check_status()
    oflags = oracle.FLAG_NO_SILU if flags & hgf.FLAG_NO_SILU else 0
    for i, (q, h, yi) in enumerate(zip(probs, hosts, y_ints)):
        ref = oracle.forward(*h, flags=oflags)
        assert np.array_equal(yi.cpu().numpy(), ref["y_int"]), (i, shapes[i])
        y, peak = ref["y"], np.abs(ref["y"]).max()
        # bf16 has eight significant bits: the result of the path, within TOL of y, is rounded by up to 2^-8 of itself
        rounding = 2.0 ** -8 * (np.abs(y) + TOL * peak) if bf16 else 0.0
        over = np.abs(q["y"].float().cpu().numpy().astype(np.float64) - y) - rounding
        assert over.max() <= TOL * peak, (i, shapes[i], over.max() / peak)
    group.close()


@pytest.mark.gpu
@pytest.mark.parametrize("base3", [False, True])
@pytest.mark.parametrize("shapes", MIXED, ids=["mixed", "two", "many", "long"])
@pytest.mark.parametrize("cap", [16, 8])
def test_group_against_oracle(hgf, shapes, base3, cap):
    """(Some of these stay on the warp MMA: the answers are the same. The next test has them all on the tensor-memory kernel.)"""
    if cap == 8 and not base3:
        pytest.skip("two-bit groups of up to eight tokens run elsewhere")
    check_group(hgf, shapes, base3, cap)


@pytest.mark.gpu
@pytest.mark.parametrize("base3,cap", [(False, 16), (True, 16), (True, 8)])
@pytest.mark.parametrize("shapes", MIXED, ids=["mixed", "two", "many", "long"])
@pytest.mark.parametrize("options", ["fp32", "bf16", "no_silu", "no_pdl"])
def test_tensor_memory_kernel_against_oracle(hgf, shapes, base3, cap, options):
    shapes = shapes + FILL
    assert most_problems(hgf, shapes, base3, cap) > 0
    flags = {"no_silu": hgf.FLAG_NO_SILU, "no_pdl": hgf.FLAG_NO_PDL}.get(options, 0)
    check_group(hgf, shapes, base3, cap, flags=flags, bf16=options == "bf16")


# Shares of several problems: from the third on, the two places of x~, H and the per-token values are used again.  Rows so long that
# the activations of two problems do not fit beside six ring stages (43 KB and more each, of 84) next to short ones, and rows that do.
MANY = {"short": ([(320, 136, 16, 1 + i % 16, 1) for i in range(700)], 16), "alternating": ([(320 if i % 2 else 3200, 40, 16, 16, 1) for i in range(620)], 16),
        "long": ([(2880 + 320 * (i % 2), 40, 16 * (i % 5), 9 + i % 8, 1) for i in range(620)], 16),
        "alternating, eight tokens": ([(320 if i % 2 else 5440, 64, 16, 8, 1) for i in range(620)], 8)}


@pytest.mark.gpu
@pytest.mark.parametrize("case,base3", [("short", False), ("short", True), ("alternating", False), ("alternating", True), ("long", False),
                                        ("long", True), ("alternating, eight tokens", True)])
def test_shares_of_many_problems(hgf, case, base3):
    shapes, cap = MANY[case]
    assert most_problems(hgf, shapes, base3, cap) >= 4
    check_group(hgf, shapes, base3, cap, variants=3)


@pytest.mark.gpu
@pytest.mark.parametrize("base3", [False, True])
def test_more_problems_on_a_cta_than_its_table_holds(hgf, base3):
    """Such a group stays on the warp MMA."""
    shapes = [(64, 16, 0, 9, 1)] * (148 * 33)
    assert most_problems(hgf, shapes, base3, 16) == 0
    check_group(hgf, shapes, base3, 16, variants=2)


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
    assert most_problems(hgf, [(q["d_in"], q["d_out"], 0, M) for q in probs], True, 16) > 0
    group = hgf.Group(probs, flags=hgf.FLAG_BASE3)
    y_ints = [torch.full(q["y"].shape, -1, dtype=torch.int32, device="cuda") for q in probs]
    for i, yi in enumerate(y_ints):
        group.debug(i, yi)
    group.forward()
    hgf.check_status()
    for i, yi in enumerate(y_ints):
        assert np.array_equal(yi.cpu().numpy(), want[i // 6])
    group.close()
