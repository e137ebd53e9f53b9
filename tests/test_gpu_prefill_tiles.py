"""prefill_gemm_kernel with tiles of 64 and of 128 tokens (prefill_tile_tokens) against the oracle: the last token and channel of a tile,
one tile and as many as there are SMs, and the first size past that."""
import numpy as np
import pytest
import torch

import oracle
from paper_2602_05269_b200 import inputs as syn

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bf16", [False, True])
@pytest.mark.parametrize("M,K,N,r", [(17, 64, 8, 16), (63, 256, 136, 32), (64, 320, 128, 0), (65, 576, 264, 64), (127, 192, 1000, 48), (129, 64, 72, 32),
                                     (64, 64, 19000, 16), (4736, 64, 256, 16), (4737, 64, 256, 32)])
def test_against_the_oracle(M, K, N, r, bf16):
    from paper_2602_05269_b200 import hgf
    W, x = syn.make_weights(N, K, config=33, layer=M), syn.make_x(M, K, config=33, layer=N)
    lora = syn.make_lora(K, N, r, config=33, layer=K) if r else (None, None, None)
    packed, gamma = hgf.pack_ternary(torch.from_numpy(W).cuda())
    dev = [None if v is None else torch.from_numpy(v).cuda() for v in lora]
    dev = [v if v is None or v.dtype == torch.float32 else v.view(torch.float16) for v in dev]
    # (rows behind y stay as they are)
    y = torch.full((M + 64, N), 7.0, dtype=torch.bfloat16 if bf16 else torch.float32, device="cuda")
    _, dbg = hgf.linear_forward(torch.from_numpy(x).view(torch.bfloat16).cuda(), packed, gamma, K, N, *dev, y=y[:M], debug=True,
                                flags=hgf.FLAG_OUT_BF16 if bf16 else 0)
    hgf.check_status()
    ref = oracle.forward(x, oracle.ternarise(W, np.float32(gamma)), np.float32(gamma), *lora)
    assert np.array_equal(dbg["y_int"].cpu().numpy(), ref["y_int"])
    tol = 6e-4 + (2.0 ** -8 if bf16 else 0.0)  # (the GEMM path's: H in fp16; bf16 rounds by up to 2^-8 of a value)
    assert np.abs(y[:M].float().cpu().numpy() - ref["y"]).max() / np.abs(ref["y"]).max() <= tol
    assert (y[M:] == 7.0).all()
