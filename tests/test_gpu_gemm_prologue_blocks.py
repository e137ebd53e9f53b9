"""gemm_prologue_kernel in blocks of eight and of sixteen warps, of 32 and of 64 tokens (short rows, so that no other kernel takes the batch), against
the oracle: codes and integer sums bit for bit, H and y within the bounds of their roundings."""
import numpy as np
import pytest
import torch

import oracle
from paper_2602_05269_b200 import inputs as syn

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,K,r,ln", [
    (17, 64, 64, False), (33, 320, 48, False), (300, 576, 64, False), (2369, 320, 64, False), (2400, 256, 64, True), (4736, 64, 48, False), (4737, 320, 48, False),
    (4737, 192, 48, True), (7000, 256, 48, False), (9476, 64, 48, False), (4740, 64, 64, False), (2369, 320, 16, False), (4737, 192, 32, False), (9480, 64, 32, False),
])
def test_against_the_oracle(M, K, r, ln):
    from paper_2602_05269_b200 import hgf
    N = 64
    W, x = syn.make_weights(N, K, config=35, layer=K), syn.make_x(M, K, config=35, layer=M)
    lora = syn.make_lora(K, N, r, config=35, layer=K) if r else (None, None, None)
    packed, gamma = hgf.pack_ternary(torch.from_numpy(W).cuda())
    T = oracle.ternarise(W, np.float32(gamma))
    dev = [None if v is None else torch.from_numpy(v).cuda() for v in lora]
    dev = [v if v is None or v.dtype == torch.float32 else v.view(torch.float16) for v in dev]
    rng = np.random.default_rng([35, M])
    w, b = (1.0 + 0.1 * rng.standard_normal(K)).astype(np.float32), (0.1 * rng.standard_normal(K)).astype(np.float32)
    fe = {"ln_weight": torch.from_numpy(w).cuda(), "ln_bias": torch.from_numpy(b).cuda()} if ln else {}
    y, dbg = hgf.linear_forward(torch.from_numpy(x).view(torch.bfloat16).cuda(), packed, gamma, K, N, *dev, debug=True, **fe)
    hgf.check_status()
    if ln:  # (the codes under the library's own statistics)
        ref = oracle.forward_ln(x, T, np.float32(gamma), w, b, 1e-5, *lora, mean=dbg["mean"].cpu().numpy(), rstd=dbg["rstd"].cpu().numpy())
    else:
        ref = oracle.forward(x, T, np.float32(gamma), *lora)
    assert np.array_equal(dbg["xq"].cpu().numpy(), ref["xq"])
    assert np.array_equal(dbg["y_int"].cpu().numpy(), ref["y_int"])
    # x A: exact products, at most K roundings of partial sums below sum |x A| (SiLU's slope is below 1.1); the activation a few ulp
    At, Bt = (v.view(np.float16).astype(np.float64) for v in lora[:2])
    bound = 1.1 * K * 2.0 ** -24 * (np.abs(syn.bf16_bits_to_f32(x)) @ np.abs(At).T) + 2.0 ** -20 * np.abs(ref["h"])
    assert np.all(np.abs(dbg["h"].cpu().numpy() - ref["h"]) <= bound)
    # y: H and gate * B rounded to fp16, 2^-11 of a value each; binary32 elsewhere
    bound = 2.0 ** -10 * 1.001 * (np.abs(ref["h"]) @ np.abs(lora[2][:, None] * Bt).T) + 1e-5 * np.abs(ref["y"]).max()
    assert np.all(np.abs(y.cpu().numpy() - ref["y"]) <= bound)
