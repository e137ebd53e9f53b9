"""rows_prologue_kernel with eight and with sixteen warps a CTA, and the batches at which launch_rows_prologue changes its mind, against the
oracle: codes and integer sums bit for bit, y within the GEMM path's tolerance."""
import ctypes

import numpy as np
import pytest
import torch

import oracle
from paper_2602_05269_b200 import inputs as syn

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,K,r,ln", [
    (17, 1088, 16, False), (448, 1024, 32, False), (465, 1024, 32, False), (465, 2112, 32, False), (577, 1024, 16, True), (1184, 1024, 32, True),
    (2049, 1024, 32, False), (2368, 1024, 48, False), (2369, 1024, 32, False), (2369, 1024, 32, True), (225, 1024, 64, False), (241, 1024, 64, False),
    (600, 1024, 64, True), (1200, 1024, 64, True), (64, 1024, 48, False), (150, 1024, 48, False), (1185, 4096, 0, True), (1185, 1024, 0, True),
])
def test_against_the_oracle(M, K, r, ln):
    from paper_2602_05269_b200 import hgf
    N = 64
    W, x = syn.make_weights(N, K, config=34, layer=K), syn.make_x(M, K, config=34, layer=M)
    lora = syn.make_lora(K, N, r, config=34, layer=K) if r else (None, None, None)
    packed, gamma = hgf.pack_ternary(torch.from_numpy(W).cuda())
    T = oracle.ternarise(W, np.float32(gamma))
    dev = [None if v is None else torch.from_numpy(v).cuda() for v in lora]
    dev = [v if v is None or v.dtype == torch.float32 else v.view(torch.float16) for v in dev]
    rng = np.random.default_rng([34, M])
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
    assert np.abs(y.cpu().numpy() - ref["y"]).max() / np.abs(ref["y"]).max() <= 6e-4


# each rank, with and without a LayerNorm: [log2 of the CTAs of a cluster, sixteen warps, shared memory for at most two CTAs an SM]
@pytest.mark.parametrize("M,K,r,ln,form", [
    (468, 2112, 16, False, [3, 0, 0]), (1186, 6336, 16, False, [2, 1, 0]), (2365, 2112, 16, False, [0, 1, 1]), (1170, 1088, 16, True, [1, 0, 1]),
    (467, 2112, 16, True, [3, 0, 0]), (2420, 3200, 16, True, [1, 0, 0]), (2427, 4160, 16, True, [1, 1, 0]), (588, 2112, 32, True, [2, 0, 1]),
    (2370, 2048, 32, True, [0, 1, 1]), (466, 2112, 32, True, [3, 0, 0]), (598, 9024, 48, False, [3, 1, 0]), (2363, 1024, 48, True, [0, 1, 1]),
    (295, 1024, 48, True, [3, 0, 1]), (1188, 1024, 48, True, [1, 0, 1]), (519, 1024, 64, False, [2, 1, 1]), (596, 7616, 64, False, [3, 0, 0]),
    (515, 1024, 64, True, [2, 1, 1]), (292, 1024, 64, True, [3, 0, 1]), (598, 7552, 64, True, [3, 0, 0]), (595, 2112, 0, True, [2, 0, 1]), (1186, 6976, 0, True, [2, 0, 0])])
def test_every_form(M, K, r, ln, form):
    from paper_2602_05269_b200 import hgf
    out = (ctypes.c_int32 * 3)()
    assert hgf.lib().hgf_internal_rows_prologue_form(M, K, 64, r, int(ln), 148, out) and [out[0], out[1], int(out[2] > 0)] == form
    test_against_the_oracle(M, K, r, ln)
