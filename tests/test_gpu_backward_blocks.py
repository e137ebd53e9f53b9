"""hgf_linear_backward at extents that are and are not multiples of 64 (operands brought by blocks of 64 rows or row by row), by single CTAs
and by pairs, against the CPU oracle; tolerance as in test_gpu_backward.py."""
import numpy as np
import pytest
import torch

import oracle
from paper_2602_05269_b200 import inputs as syn
from test_backward_thin_cpu import trace

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


def _arguments(M, K, N, r):
    from paper_2602_05269_b200 import hgf
    g = torch.Generator(device="cuda")
    g.manual_seed(M + 7 * K + 13 * N + r)
    rand = lambda *shape: torch.randn(shape, generator=g, device="cuda")  # noqa: E731
    x, dy = rand(M, K).to(torch.bfloat16), rand(M, N).to(torch.bfloat16)
    packed, gamma = hgf.pack_ternary(0.02 * rand(N, K))
    At, Bt, gate = (K ** -0.5 * rand(r, K)).half(), (r ** -0.5 * rand(N, r)).half(), rand(N).abs()
    return x, packed, gamma, K, N, dy, At, Bt, gate


def _exact(x, packed, gamma, K, N, dy, At, Bt, gate):
    """The four gradients that do not take quantised activations, in 64 bits."""
    from paper_2602_05269_b200 import hgf
    z = x.double() @ At.double().t()
    s = torch.sigmoid(z)
    G = dy.double().t() @ (z * s)
    dz = ((dy.double() * gate.double()) @ Bt.double()) * (s * (1 + z * (1 - s)))
    ref = {"dx": gamma * (dy.double() @ hgf.unpack_ternary(packed, N, K).double()) + dz @ At.double(), "dAt": dz.t() @ x.double(),
           "dBt": gate.double()[:, None] * G, "dgate": (G * Bt.double()).sum(1)}
    return ref


# dW's launch takes dH and G along, and dA is a launch of its own whose contraction is split often enough to fill the room for partial sums
@pytest.mark.parametrize("without_dx,M,K,N,r", [(False, 4096, 2112, 2048, 32), (False, 2656, 3456, 3456, 16), (False, 2500, 2112, 512, 48), (False, 4096, 2176, 3072, 64),
                                                (True, 3072, 3072, 3072, 32), (True, 4096, 2560, 2560, 16), (True, 2560, 2560, 2560, 48)])
def test_partial_sums_of_two_products_at_a_time(without_dx, M, K, N, r):
    """Tolerance as in test_gpu_backward.py, 2^-9 of a typical term, here in the 2-norm: within 5e-3 of the gradient's."""
    from paper_2602_05269_b200 import hgf
    args = _arguments(M, K, N, r)
    ref = _exact(*args)
    want = ("dW", "dAt", "dBt", "dgate") if without_dx else ("dx", "dW", "dAt", "dBt", "dgate")
    assert trace(hgf.lib(), M, K, N, r, want)[2][::4] == [2, 0]
    got = hgf.linear_backward(*args, want=want)
    hgf.check_status()
    for n in ref:
        if n in got:
            err = float((got[n].double() - ref[n]).norm() / ref[n].norm())
            assert err <= 5e-3, f"{n}: {err:.3e}"


# dW's launch takes dH and G along, dX's takes dA, or not; asked for without dW and dx the same products are launches of their own
@pytest.mark.parametrize("M,K,N,r", [(8192, 2048, 5632, 32), (2048, 2048, 2048, 32), (700, 1024, 3000, 32), (8000, 768, 1536, 64), (4096, 4096, 4096, 16),
                                     (1500, 3200, 2000, 64), (512, 2048, 2048, 48), (5000, 4160, 1000, 32)])
def test_a_gradient_has_the_same_bits_whichever_others_are_asked_for(M, K, N, r):
    from paper_2602_05269_b200 import hgf
    args = _arguments(M, K, N, r)
    got = hgf.linear_backward(*args)
    for want in (("dBt", "dgate"), ("dAt",), ("dx",), ("dW",), ("dx", "dAt"), ("dW", "dAt")):
        alone = hgf.linear_backward(*args, want=want)
        for n in want:
            assert torch.equal(alone[n], got[n]), f"{n} by itself as {want}: {(alone[n] - got[n]).norm() / got[n].norm():.1e} apart"
    hgf.check_status()


# [thin products, half tiles, c_idle, c_busy] of dW's launch and of dX's: pairs that go from a tile to a piece, that take several pieces, and that go
# from half a tile to a piece; parts of one partial sum and of several, a last one that is shorter
@pytest.mark.parametrize("M,K,N,r,rides", [
    (466, 512, 520, 16, [2, 0, 1, 0, 1, 0, 1, 0]), (1102, 640, 4104, 48, [2, 0, 1, 1, 1, 0, 1, 0]), (2314, 576, 4560, 32, [2, 0, 2, 1, 1, 0, 1, 0]),
    (577, 2304, 2904, 64, [2, 68, 0, 1, 1, 0, 1, 0]), (1426, 1280, 4784, 16, [2, 42, 1, 1, 1, 0, 1, 0]), (1681, 2304, 2720, 32, [2, 50, 2, 0, 1, 0, 1, 0]),
    (2063, 2048, 3128, 48, [2, 60, 2, 1, 0, 0, 0, 0]), (2200, 4864, 936, 64, [2, 4, 1, 0, 1, 46, 2, 1]), (1835, 3328, 560, 16, [2, 0, 1, 0, 1, 60, 0, 1]),
    (3189, 2048, 2600, 32, [2, 28, 2, 0, 1, 60, 2, 0]), (5777, 512, 512, 64, [2, 0, 1, 0, 0, 0, 0, 0]), (408, 4992, 792, 32, [0, 0, 0, 0, 1, 0, 1, 0]),
    (1774, 4864, 600, 48, [2, 0, 1, 0, 1, 0, 2, 1]), (3072, 3072, 3072, 16, [2, 0, 1, 1, 1, 0, 0, 1])])
def test_pairs_that_take_tiles_and_pieces(M, K, N, r, rides):
    """Against 64 bits (tolerance as above); dW and what rides beside it are the bits that they are without each other."""
    from paper_2602_05269_b200 import hgf
    assert trace(hgf.lib(), M, K, N, r)[2] == rides
    args = _arguments(M, K, N, r)
    ref, got = _exact(*args), hgf.linear_backward(*args)
    for n in ref:
        err = float((got[n].double() - ref[n]).norm() / ref[n].norm())
        assert err <= 5e-3, f"{n}: {err:.3e}"
    assert torch.equal(got["dW"], hgf.linear_backward(*args[:6], want=("dW",))["dW"])
    for want in (("dBt", "dgate"), ("dAt",), ("dx",)):
        alone = hgf.linear_backward(*args, want=want)
        assert all(torch.equal(alone[n], got[n]) for n in want), want
    hgf.check_status()
