"""Base-3 weights on the GEMM path (repack_b3_kernel): the same bits as the call on two-bit weights, at the edges of both tile widths."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K,N", [(64, 8), (256, 24), (320, 16), (384, 136), (640, 40), (1280, 72), (1344, 256), (11008, 128)])
def test_same_bits_as_on_two_bit_weights(K, N):
    from paper_2602_05269_b200 import hgf
    g = torch.Generator(device="cuda").manual_seed(K + N)
    W = torch.randn((N, K), generator=g, device="cuda") * 0.02
    x = torch.randn((33, K), generator=g, device="cuda").to(torch.bfloat16)
    y2 = hgf.linear_forward(x, *hgf.pack_ternary(W), K, N)
    # (a workspace full of other bits: words of padding columns are written too)
    ws = torch.full((hgf.workspace_bytes(33, K, N, 0, hgf.FLAG_BASE3),), 0xff, dtype=torch.uint8, device="cuda")
    y3 = hgf.linear_forward(x, *hgf.pack_ternary(W, base3=True), K, N, workspace=ws, flags=hgf.FLAG_BASE3)
    hgf.check_status()
    assert torch.equal(y2, y3)
