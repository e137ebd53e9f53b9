"""hgf_linear_backward at extents that are and are not multiples of 64 (operands brought by blocks of 64 rows or row by row), by single CTAs
and by pairs, against the CPU oracle; tolerance as in test_gpu_backward.py."""
import numpy as np
import pytest
import torch

import oracle
from paper_2602_05269_b200 import inputs as syn

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,K,N,r", [(700, 448, 320, 16), (640, 1088, 576, 48), (700, 448, 328, 64), (448, 320, 264, 0), (1000, 576, 1344, 32), (96, 192, 448, 32)])
def test_gradients(M, K, N, r):
    from paper_2602_05269_b200 import hgf
    L = syn.make_layer(syn.LayerShape("bw", K, N, max(r, 16)), M, config=25, layer=M + N)
    dev = lambda a, t=None: torch.from_numpy(np.ascontiguousarray(a)).cuda() if t is None else torch.from_numpy(np.ascontiguousarray(a)).view(t).cuda()  # noqa: E731
    packed, gamma = hgf.pack_ternary(dev(L["W"]))
    dy = syn.f32_to_bf16_bits(np.random.default_rng([73, M]).standard_normal((M, N)).astype(np.float32))
    lora = (L["At"], L["Bt"], L["gate"]) if r else (None, None, None)
    got = hgf.linear_backward(dev(L["x"], torch.bfloat16), packed, gamma, K, N, dev(dy, torch.bfloat16),
                              *((dev(lora[0], torch.float16), dev(lora[1], torch.float16), dev(lora[2])) if r else ()))
    hgf.check_status()
    ref = oracle.backward(L["x"], oracle.ternarise(L["W"], np.float32(gamma)), gamma, dy, *lora)
    for n in ref:
        err = np.abs(got[n].cpu().numpy().astype(np.float64) - ref[n]).max() / np.abs(ref[n]).max()
        assert err <= 1e-2, f"{n}: normalised error {err:.3e}"
