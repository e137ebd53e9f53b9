"""Two-bit packing, word for word: codes of the oracle's threshold under the scale returned, code 1 in the padding, the scale the rounded mean."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,K", [(1, 64), (16, 256), (17, 320), (15, 704), (333, 1088), (2049, 256), (1030, 4096), (2500, 2112)])
def test_words(N, K):
    from paper_2602_05269_b200 import hgf
    rng = np.random.default_rng([6, N, K])
    W = (rng.standard_normal((N, K)) * 0.02).astype(np.float32)
    W[N // 2, :64] = 0.0
    packed, gamma = hgf.pack_ternary(torch.from_numpy(W).cuda())
    mean = np.abs(W.astype(np.float64)).mean()
    assert abs(gamma - mean) <= 2.0 ** -23 * mean  # (sums in double, one rounding to binary32)
    rows, cols = -(-N // 16) * 16, -(-K // 256) * 256
    T = np.zeros((rows, cols), np.int64)
    T[:N, :K] = oracle.ternarise(W, np.float32(gamma))
    codes = (T + 1).astype(np.uint32)
    # [row tile][column tile][row][word][j][b]: weight 4 j + b of a word in bits 8 b + 2 j
    c = codes.reshape(rows // 16, 16, cols // 256, 16, 4, 4).transpose(0, 2, 1, 3, 4, 5)
    shift = (8 * np.arange(4)[None, :] + 2 * np.arange(4)[:, None]).astype(np.uint32)
    words = (c << shift).sum(axis=(-1, -2), dtype=np.uint32).reshape(-1)
    assert np.array_equal(packed.cpu().numpy().view(np.uint32), words)


def test_no_scale():
    """All weights zero: scale 0, code 1 everywhere.  A NaN: every comparison with it fails, code 1 everywhere, too."""
    from paper_2602_05269_b200 import hgf
    W = torch.zeros((33, 192), device="cuda")
    packed, gamma = hgf.pack_ternary(W)
    assert gamma == 0.0 and bool((packed == 0x55).all())
    W = torch.randn((33, 192), device="cuda")
    W[5, 7] = float("nan")
    packed, gamma = hgf.pack_ternary(W)
    assert gamma != gamma and bool((packed == 0x55).all())
