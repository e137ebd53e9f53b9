"""Parity of hgf_linear_backward (straight-through backward pass of the layer, paper Section 2.2) against
the CPU oracle through the C ABI.

Tolerance: the matrix products take bf16 operands with fp32 accumulation (the paper trains under bf16
autocast).  x~ and the ternary codes are exact in bf16; dY scaled by gamma_x / 127 or by the gate, A, B, H and
dZ are each rounded once (relative 2^-9), and a sum of such terms with random signs keeps a relative error of
about 2^-9 of its typical term: every gradient must be within 1e-2 of the oracle's, normalised by max|ref|."""
import numpy as np
import pytest
import torch

import oracle
from paper_2602_05269_b200 import inputs as syn

pytestmark = pytest.mark.gpu

TOL = 1e-2


@pytest.fixture(scope="module")
def hgf():
    assert torch.cuda.is_available(), "these tests need a CUDA device"
    from paper_2602_05269_b200 import hgf as binding
    binding.lib()
    torch.cuda.set_device(0)
    return binding


def dev(a, dtype=None):
    t = torch.from_numpy(np.ascontiguousarray(a))
    return (t.view(dtype) if dtype is not None else t).cuda()


def check(hgf, M, K, N, r, *, layer, flags=0, lora=True, want=None):
    L = syn.make_layer(syn.LayerShape("bw", K, N, max(r, 16)), M, config=24, layer=layer)
    packed, gamma = hgf.pack_ternary(dev(L["W"]))
    T = oracle.ternarise(L["W"], np.float32(gamma))
    dy = syn.f32_to_bf16_bits(np.random.default_rng([72, layer]).standard_normal((M, N)).astype(np.float32))
    use = lora and r > 0
    got = hgf.linear_backward(dev(L["x"], torch.bfloat16), packed, gamma, K, N, dev(dy, torch.bfloat16),
                              dev(L["At"], torch.float16) if use else None, dev(L["Bt"], torch.float16) if use else None,
                              dev(L["gate"]) if use else None, flags=flags, want=want)
    torch.cuda.synchronize()
    oflags = oracle.FLAG_NO_SILU if flags & hgf.FLAG_NO_SILU else 0
    ref = oracle.backward(L["x"], T, gamma, dy, L["At"] if use else None, L["Bt"] if use else None, L["gate"] if use else None,
                          flags=oflags)
    names = [n for n in ref if want is None or n in want]
    assert set(n for n in got if not n.startswith("_")) == set(names)
    for n in names:
        g = got[n].cpu().numpy().astype(np.float64)
        err = np.abs(g - ref[n]).max() / np.abs(ref[n]).max()
        assert err <= TOL, f"{n}: normalised error {err:.3e} (M={M} K={K} N={N} r={r})"


@pytest.mark.parametrize("M,K,N,r", [(64, 256, 128, 16), (200, 512, 264, 32), (300, 1024, 1000, 48), (129, 448, 72, 64),
                                     (17, 64, 8, 16), (512, 2048, 2048, 32)])
def test_all_gradients(hgf, M, K, N, r):
    check(hgf, M, K, N, r, layer=M)


def test_pure_ternary_layer_no_silu_and_selected_outputs(hgf):
    check(hgf, 150, 512, 256, 0, layer=1, lora=False)
    check(hgf, 150, 512, 256, 32, layer=2, flags=hgf.FLAG_NO_SILU)
    check(hgf, 150, 512, 256, 32, layer=3, want=("dW",))
    check(hgf, 150, 512, 256, 32, layer=4, want=("dx", "dgate"))


def test_more_tiles_than_sms_with_a_ragged_last_round(hgf):
    """dW of 2560 x 2048 and dX of 2560 x 2048 are 160 output tiles of 128 x 256 each: more than the SMs of the
    part, with a last round of the persistent schedule that the kernel works as twice as many half-width tiles.
    The small other extent keeps the oracle affordable."""
    check(hgf, 64, 2048, 2560, 32, layer=6)    # dW [2560][2048]
    check(hgf, 2560, 2048, 64, 32, layer=7)    # dX [2560][2048], with the low-rank term in the same contraction
    check(hgf, 2560, 2048, 64, 0, layer=8, lora=False)


def test_decode_sized_batch(hgf):
    check(hgf, 4, 2048, 512, 32, layer=5)


def test_rejects_bad_arguments(hgf):
    x = torch.zeros((8, 256), dtype=torch.bfloat16, device="cuda")
    packed = torch.zeros(hgf.packed_bytes(60, 256), dtype=torch.uint8, device="cuda")
    dy = torch.zeros((8, 60), dtype=torch.bfloat16, device="cuda")
    with pytest.raises(hgf.HgfError) as e:          # d_out must be a multiple of 8
        hgf.linear_backward(x, packed, 1.0, 256, 60, dy)
    assert e.value.status == 2


@pytest.mark.parametrize("M,K,N,r", [(40, 4096, 64, 16), (33, 4160, 64, 16), (9, 2112, 72, 32), (70, 2048, 40, 16)])
def test_row_lengths_of_the_quantiser(hgf, M, K, N, r):
    """Rows at the limits of what a warp holds in registers (2048, 4096 columns) and just past them."""
    check(hgf, M, K, N, r, layer=K)


@pytest.mark.parametrize("M,K,N,r", [(40, 192, 136, 16), (257, 320, 264, 64), (256, 256, 256, 32), (1, 192, 136, 0), (130, 2112, 384, 48)])
def test_outputs_just_past_one_tile(hgf, M, K, N, r):
    """Outputs just past 128 rows and columns with a short contraction (single CTAs): ragged tiles, a contraction of one element."""
    check(hgf, M, K, N, r, layer=M + 500, lora=r > 0)


# contractions that pairs take: dW contracts over M, dX over N (and r)
@pytest.mark.parametrize("M,K,N,r", [(440, 192, 136, 16), (700, 320, 264, 64), (768, 256, 256, 32), (641, 192, 136, 0), (136, 192, 640, 16),
                                     (257, 320, 648, 64), (256, 256, 768, 0), (650, 2112, 704, 48)])
def test_tiles_of_cta_pairs(hgf, M, K, N, r):
    """Outputs just past 128 rows and columns (the second CTA of a pair has 8 rows, or none), exact 256 x 256 tiles, a contraction that
    ends inside a block, column tiles that end inside the second CTA's half."""
    check(hgf, M, K, N, r, layer=M + 500, lora=r > 0)


def _close(got, a, b, alpha=1.0):
    """got = alpha a b in fp32 against 64 bits: each of the C products is exact in fp32; an addition in the tensor core's accumulator may
    cut off instead of rounding and align its products first, so it is charged 2^-22 of the sum of magnitudes."""
    a, b = a.double(), b.double()
    bound = (a.shape[1] + 2) * 2.0 ** -22 * abs(alpha) * (a.abs() @ b.abs())
    err = (got.double() - alpha * (a @ b)).abs()
    assert bool((err <= bound).all()), float((err / bound.clamp_min(1e-30)).max())


@pytest.mark.parametrize("C,I,J", [(648, 4088, 4160), (640, 4096, 4096), (648, 3592, 4096)])
def test_cta_pairs_with_many_tiles_each(hgf, C, I, J):
    """Every pair of CTAs takes at least three output tiles, so accumulators are handed back between the two CTAs and used again:
    dW (both operands with the contraction outside) and dX (the first one with it inside), ragged in both extents, and last rounds
    of whole and of half tiles."""
    assert hgf.lib().hgf_internal_tc_pairs_pay(I, J, C, 148, 74) == 1
    g = torch.Generator(device="cuda")
    g.manual_seed(C + I)
    W = torch.randn((I, J), generator=g, device="cuda")
    packed, gamma = hgf.pack_ternary(W)
    x = torch.randn((C, J), generator=g, device="cuda").to(torch.bfloat16)
    dy = torch.randn((C, I), generator=g, device="cuda").to(torch.bfloat16)
    got = hgf.linear_backward(x, packed, gamma, J, I, dy, want=("dW",))["dW"]
    xq, gx, _ = hgf.act_quant(x)
    xd = (xq.float() * (gx * (1.0 / 127.0))[:, None]).to(torch.bfloat16)
    _close(got, dy.t(), xd)
    packed, gamma = hgf.pack_ternary(W[:C])
    T = hgf.unpack_ternary(packed, C, J)
    x = torch.randn((I, J), generator=g, device="cuda").to(torch.bfloat16)
    dy = torch.randn((I, C), generator=g, device="cuda").to(torch.bfloat16)
    _close(hgf.linear_backward(x, packed, gamma, J, C, dy, want=("dx",))["dx"], dy, T, gamma)
    hgf.check_status()
