"""Packing calls in flight at the same time, from more threads than the library has scratch slots, each on a stream
of its own: every call's codes and scale are those of the same matrix packed alone and of the oracle's threshold."""
from concurrent.futures import ThreadPoolExecutor

import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("base3", [False, True])
def test_packing_from_many_threads(base3):
    from paper_2602_05269_b200 import hgf
    hgf.lib()
    # one weight tile, ragged tiles, fewer and more rows than the partial sums of the scale cover
    shapes = [(1, 64), (16, 256), (24, 320), (40, 512), (333, 1088), (700, 2048), (1024, 4096)]
    rng = np.random.default_rng(5)
    mats = [(rng.standard_normal(shapes[i % len(shapes)]) * 0.02).astype(np.float32) for i in range(48)]
    dev = [torch.from_numpy(W).cuda() for W in mats]
    alone = [hgf.pack_ternary(W, base3=base3) for W in dev]
    torch.cuda.synchronize()

    def pack(W):
        with torch.cuda.stream(torch.cuda.Stream()):
            return hgf.pack_ternary(W, base3=base3)

    with ThreadPoolExecutor(24) as pool:
        together = list(pool.map(pack, dev))
    torch.cuda.synchronize()
    for W, (p0, g0), (p1, g1) in zip(mats, alone, together):
        assert g0 == g1 and torch.equal(p0, p1)
        assert abs(g0 - float(oracle.gamma_w(W))) <= g0 * 2.0 ** -23
        T = oracle.ternarise(W, np.float32(g0))
        assert np.array_equal(p0.cpu().numpy(), oracle.pack_b3(T) if base3 else oracle.pack(T))
