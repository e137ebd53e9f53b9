"""The clustered prologue of the GEMM path at the edges of its split, against the oracle: one token past the decode path,
blocks of sixteen tokens that are not full, slices of unequal width and CTAs of a cluster that get none, every rank, with and
without the LayerNorm, subnormal and constant tokens.  Codes, scales and int32 accumulators bit for bit (behind a LayerNorm
under the library's own statistics), H to fp32 summation (K 2^-24 of the sum of magnitudes, here below 1e-5 of the largest),
y to the GEMM path's 6e-4 (H enters in fp16)."""
import numpy as np
import pytest
import torch

import oracle
from paper_2602_05269_b200 import inputs as syn

pytestmark = pytest.mark.gpu


def dev(a, dtype=None):
    t = torch.from_numpy(np.ascontiguousarray(a))
    return (t.view(dtype) if dtype is not None else t).cuda()


@pytest.mark.parametrize("ln", [False, True])
@pytest.mark.parametrize("M,K,r", [(17, 1024, 16), (31, 1088, 32), (33, 5632, 48), (64, 1024, 0), (95, 1600, 64), (200, 2048, 32), (513, 1216, 16),
                                   (1100, 2112, 64), (2048, 1024, 32), (70, 11008, 64), (130, 192, 0),
                                   (1024, 768, 0), (1100, 576, 0), (1300, 576, 0), (1920, 64, 0), (1150, 1024, 64), (1184, 1024, 64), (2048, 1088, 64), (570, 1024, 48), (1300, 1024, 16)])
def test_rows_prologue(M, K, r, ln):
    from paper_2602_05269_b200 import hgf
    N = 40
    L = syn.make_layer(syn.LayerShape("rows", K, N, max(r, 16)), M, config=21, layer=M + K)
    At, Bt, gate = (L["At"], L["Bt"], L["gate"]) if r else (None, None, None)
    x = L["x"].copy()
    x[1] = 0                                                             # an all-zero token
    x[2] = syn.f32_to_bf16_bits(np.full(K, 3.0, np.float32))             # a constant one
    x[3, : K // 2] = 0x0001                                              # subnormals beside ordinary values
    packed, gamma = hgf.pack_ternary(dev(L["W"]))
    T = oracle.ternarise(L["W"], np.float32(gamma))
    rng = np.random.default_rng([33, M])
    w, b = (1.0 + 0.2 * rng.standard_normal(K)).astype(np.float32), (0.1 * rng.standard_normal(K)).astype(np.float32)
    fe = {"ln_weight": dev(w), "ln_bias": dev(b), "eps": 1e-5} if ln else {}
    y, dbg = hgf.linear_forward(dev(x, torch.bfloat16), packed, gamma, K, N, None if not r else dev(At, torch.float16),
                                None if not r else dev(Bt, torch.float16), None if not r else dev(gate), debug=True, **fe)
    hgf.check_status()
    if ln:
        mean, rstd = dbg["mean"].cpu().numpy(), dbg["rstd"].cpu().numpy()
        mean_o, rstd_o = oracle.ln_stats(x, 1e-5)
        assert np.all(np.abs(mean - mean_o) <= 2e-7 * np.sqrt(1.0 / rstd_o ** 2 + mean_o ** 2)) and np.all(np.abs(rstd / rstd_o - 1) <= 3e-7)
        ref = oracle.forward_ln(x, T, gamma, w, b, 1e-5, At, Bt, gate, mean=mean, rstd=rstd)
    else:
        ref = oracle.forward(x, T, gamma, At, Bt, gate)
    assert np.array_equal(dbg["xq"].cpu().numpy(), ref["xq"]) and np.array_equal(dbg["gamma_x"].cpu().numpy(), ref["gamma_x"])
    assert np.array_equal(dbg["y_int"].cpu().numpy(), ref["y_int"])
    if r:
        assert np.abs(dbg["h"].cpu().numpy() - ref["h"]).max() <= 1e-5 * np.abs(ref["h"]).max()
    assert np.abs(y.cpu().numpy() - ref["y"]).max() <= 6e-4 * np.abs(ref["y"]).max()


@pytest.mark.parametrize("bf16", [False, True])
@pytest.mark.parametrize("M,K,N,r", [(17, 11008, 1024, 16), (100, 11008, 1000, 0), (64, 5632, 2048, 32), (129, 5632, 1032, 64), (512, 5632, 2048, 32),
                                     (300, 4096, 3000, 48), (2000, 4160, 512, 32), (33, 4288, 128, 16), (128, 11008, 4096, 64)])
def test_contraction_divided_over_a_cluster(M, K, N, r, bf16):
    """Few output tiles and a long K: two, four and eight CTAs a tile, uneven shares of the K blocks, tiles that end inside
    a token chunk and inside a channel quarter.  The int32 sums are exact (against float64 products of the same codes), y is the
    dequantised sum plus the correction in float64 (6e-4: H enters in fp16; half a bf16 ulp more in bf16)."""
    from paper_2602_05269_b200 import hgf
    g = torch.Generator(device="cuda").manual_seed(M + K)
    rn = lambda shape, std=1.0: torch.randn(shape, generator=g, device="cuda") * std  # noqa: E731
    packed, gamma = hgf.pack_ternary(rn((N, K), 0.02))
    x = rn((M, K)).bfloat16()
    At, Bt, gate = (rn((r, K), K ** -0.5).half(), rn((N, r), r ** -0.5).half(), torch.rand(N, generator=g, device="cuda")) if r else (None,) * 3
    y, dbg = hgf.linear_forward(x, packed, gamma, K, N, At, Bt, gate, debug=True, flags=hgf.FLAG_OUT_BF16 if bf16 else 0)
    hgf.check_status()
    T = hgf.unpack_ternary(packed, N, K).double()
    y_int = dbg["xq"].double() @ T.T
    assert torch.equal(dbg["y_int"].double(), y_int)
    ref = y_int * dbg["gamma_x"].double()[:, None] * gamma / 127.0
    if r:
        z = x.double() @ At.double().T
        ref = ref + (z * torch.sigmoid(z)) @ Bt.double().T * gate.double()
    assert float((y.double() - ref).abs().max()) <= (6e-4 + (2.0 ** -8 if bf16 else 0.0)) * float(ref.abs().max())
