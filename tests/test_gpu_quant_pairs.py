"""Rounding two values an instruction (quant_rows_kernel, round_rows_kernel) against one at a time (quant_kernel): the same bytes, for ordinary
rows and for ties, zeros, magnitudes whose product with 127 overflows, infinities and NaN."""
import numpy as np
import pytest
import torch

from paper_2602_05269_b200 import inputs as syn

pytestmark = pytest.mark.gpu


def rows(M, K):
    x = syn.bf16_bits_to_f32(syn.make_x(M, K, config=41, layer=K))
    x[0, :3] = [1216.0, 608.0, -608.0]     # 63.5, -63.5: ties
    x[1] = 0.0
    x[2, :4] = [127.0, 2.5, -3.5, 6.5]
    x[3, :2] = [3.0e38, -3.0e38]
    x[4] *= 1e-30
    x[5, 7] = np.inf
    x[6, :2] = [-np.inf, np.inf]
    x[7, K - 1] = np.nan
    return syn.f32_to_bf16_bits(x)


@pytest.mark.parametrize("M,K,r", [(256, 64, 0), (259, 2048, 0), (256, 4096, 0), (65, 4160, 0), (2385, 2048, 16), (4097, 1088, 32)])
def test_same_codes_as_one_row_at_a_time(M, K, r):
    from paper_2602_05269_b200 import hgf
    x = torch.from_numpy(rows(M, K)).view(torch.bfloat16).cuda()
    if r:  # (the codes of the whole layer call; its rounding is a launch of its own from 8 MB of x on)
        W, lora = syn.make_weights(16, K, config=41, layer=K), syn.make_lora(K, 16, r, config=41, layer=K)
        packed, gamma = hgf.pack_ternary(torch.from_numpy(W).cuda())
        dev = [torch.from_numpy(v).cuda() for v in lora]
        dev = [v if v.dtype == torch.float32 else v.view(torch.float16) for v in dev]
        _, dbg = hgf.linear_forward(x, packed, gamma, K, 16, *dev, debug=True)
        xq = dbg["xq"]
    else:
        xq, _, row_sum = hgf.act_quant(x)
        assert torch.equal(row_sum, xq.sum(dim=1, dtype=torch.int32))
    for m in list(range(10)) + [M // 2, M - 1]:
        one = hgf.act_quant(x[m:m + 1])[0]
        assert torch.equal(xq[m:m + 1], one), m
    hgf.check_status()
