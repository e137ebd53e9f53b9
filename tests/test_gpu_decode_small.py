"""The one-launch decode path against the two-launch path (the same call's two phases run apart) on the same inputs:
codes, scales and int32 accumulators bit for bit; y within 2e-5 of its largest value (the sums of x A are added in
another order in fp32, at most K 2^-24 relative, and both paths carry H to 2^-22).  Sizes at the edges of its split: one
column tile and less, ragged row tiles, fewer row tiles than CTAs, more warps than column tiles, every rank."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu

SHAPES = [(1, 64, 1, 16), (1, 192, 40, 0), (16, 256, 17, 64), (9, 320, 1000, 48), (2, 512, 512, 16), (1, 2048, 2048, 32),
          (4, 2048, 24, 32), (3, 1600, 1544, 64), (1, 5632, 2048, 32), (7, 1088, 4096, 0), (16, 512, 5632, 32), (2, 4096, 300, 32)]


@pytest.fixture(scope="module")
def hgf():
    from paper_2602_05269_b200 import hgf as binding
    binding.lib()
    return binding


def layer(hgf, M, K, N, r, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    rn = lambda shape, std=1.0: torch.randn(shape, generator=g, device="cuda") * std  # noqa: E731
    packed, gamma = hgf.pack_ternary(rn((N, K), 0.02))
    x = rn((M, K))
    x[:, : K // 50] *= 20.0
    c = {"At": None, "Bt": None, "gate": None}
    if r:
        c = {"At": rn((r, K), K ** -0.5).half(), "Bt": rn((N, r), r ** -0.5).half(), "gate": torch.rand(N, generator=g, device="cuda")}
    return x.bfloat16(), packed, gamma, c


def host(t):
    """A device tensor as the oracle takes it: 16-bit floats by their bit patterns, None as it is."""
    if t is None:
        return None
    return t.cpu().view(torch.int16).numpy().view(np.uint16) if t.dtype in (torch.bfloat16, torch.float16) else t.cpu().numpy()


@pytest.mark.parametrize("M,K,N,r", SHAPES)
def test_one_launch_equals_two(hgf, M, K, N, r):
    x, packed, gamma, c = layer(hgf, M, K, N, r, 7 * K + N + M)
    ws = torch.zeros(hgf.workspace_bytes(M, K, N, r), dtype=torch.uint8, device="cuda")
    kw = dict(workspace=ws, debug=True, **c)
    before = hgf.launch_count()
    y1, d1 = hgf.linear_forward(x, packed, gamma, K, N, **kw)
    assert hgf.launch_count() - before == 1, "this size is meant for the one-launch path"
    _, d2 = hgf.linear_forward(x, packed, gamma, K, N, phases=1, **kw)
    y2, d3 = hgf.linear_forward(x, packed, gamma, K, N, phases=2, **kw)
    hgf.check_status()
    assert torch.equal(d1["xq"], d2["xq"]) and torch.equal(d1["gamma_x"], d2["gamma_x"]) and torch.equal(d1["y_int"], d3["y_int"])
    assert float((y1 - y2).abs().max()) <= 2e-5 * float(y2.abs().max())
    # what a whole call leaves in the workspace serves a contraction run on its own, with and without the debug H
    for debug in (True, False):
        kw["debug"] = debug
        ws.fill_(0x5a)
        hgf.linear_forward(x, packed, gamma, K, N, **kw)
        y3 = hgf.linear_forward(x, packed, gamma, K, N, phases=2, **kw)
        y3 = y3[0] if debug else y3
        assert float((y3 - y1).abs().max()) <= 2e-5 * float(y1.abs().max())


@pytest.mark.parametrize("M,K", [(1, 64), (2, 2048), (4, 1024), (12, 320)])
@pytest.mark.parametrize("r", [0, 32])
def test_layernorm_group_equals_its_layers(hgf, M, K, r):
    """A group of three projections of one x, each behind its LayerNorm, in one launch: against the oracle, codes, scales
    and int32 accumulators bit for bit under the library's own statistics; and against the same group's two phases."""
    g = torch.Generator(device="cuda").manual_seed(K + M)
    problems = []
    x = (torch.randn((M, K), generator=g, device="cuda") * 3 + 1).bfloat16()
    for i, N in enumerate((64, 208, 1024)):
        _, packed, gamma, c = layer(hgf, M, K, N, r, 100 * K + i)
        if r:
            c["gate"] = c["gate"][: -(-N // 16)].contiguous()
        stat = {n: torch.zeros(M, device="cuda") for n in ("mean_out", "rstd_out")}
        problems.append({"x": x, "d_in": K, "d_out": N, "packed": packed, "gamma": gamma, "y": torch.empty((M, N), device="cuda"), "gate_group": 16,
                         "eps": 1e-5, "ln_weight": 1 + 0.1 * torch.randn(K, generator=g, device="cuda"), "ln_bias": 0.1 * torch.randn(K, generator=g, device="cuda"),
                         **stat, **c})
    group = hgf.Group(problems)
    yi = [torch.empty((M, p["d_out"]), dtype=torch.int32, device="cuda") for p in problems]
    views = [group.debug(i, yi[i]) for i in range(3)]
    before = hgf.launch_count()
    group.forward()
    assert hgf.launch_count() - before == 1
    hgf.check_status()
    y1, yi1, xq1 = [p["y"].clone() for p in problems], [t.clone() for t in yi], [v["xq"].clone() for v in views]
    xd = x.double()
    mean, var = xd.mean(1), xd.var(1, unbiased=False)
    for p, view, i, y in zip(problems, views, yi, y1):
        assert float((p["mean_out"].double() - mean).abs().max()) <= 2e-7 * float(xd.square().mean().sqrt())
        assert float((p["rstd_out"].double() * (var + 1e-5).sqrt() - 1).abs().max()) <= 3e-7
        T = hgf.unpack_ternary(p["packed"], p["d_out"], K).cpu().numpy()
        ref = oracle.forward_ln(host(x), T, p["gamma"], host(p["ln_weight"]), host(p["ln_bias"]), 1e-5, host(p["At"]), host(p["Bt"]),
                                host(p["gate"]), gate_group=16, mean=host(p["mean_out"]), rstd=host(p["rstd_out"]))
        assert np.array_equal(host(view["xq"]), ref["xq"]) and np.array_equal(host(view["gamma_x"]), ref["gamma_x"])
        assert np.array_equal(host(i), ref["y_int"])
        assert np.abs(host(y) - ref["y"]).max() <= 2e-5 * np.abs(ref["y"]).max()
    group.forward_phases(1)
    group.forward_phases(2)
    hgf.check_status()
    for p, a, b, c, v, i in zip(problems, y1, yi1, xq1, views, yi):
        # (the statistics are rounded to binary32 from two differently summed doubles: a last-bit tie may move a code)
        assert float((v["xq"] != c).float().mean()) <= 1e-3 and float((i != b).float().mean()) <= 0.02
        assert float((p["y"] - a).abs().max()) <= 2e-3 * float(a.abs().max())
    group.close()


@pytest.mark.parametrize("M,K,N,r", [(1, 2048, 2048, 32), (4, 512, 512, 16), (16, 320, 1000, 64)])
def test_gate_written_by_the_launch_before(hgf, M, K, N, r):
    """The gates are the outputs of a layer call still pending on the stream, which lets the next launch start early: the
    result is that of the same gates at rest."""
    x, packed, gamma, c = layer(hgf, M, K, N, r, 5 * K + r)
    xg, pg, gg, cg = layer(hgf, 1, 512, N, 16, 11)
    gates = torch.empty((1, N), device="cuda")

    def pair():
        hgf.linear_forward(xg, pg, gg, 512, N, y=gates, **cg)
        return hgf.linear_forward(x, packed, gamma, K, N, c["At"], c["Bt"], gates[0])

    pair()
    torch.cuda.synchronize()
    ref = hgf.linear_forward(x, packed, gamma, K, N, c["At"], c["Bt"], gates[0])
    for _ in range(20):
        gates.fill_(float("nan"))
        assert torch.equal(pair(), ref)
    hgf.check_status()


@pytest.mark.parametrize("n", [3, 30])
def test_captured_group_follows_the_debug_buffer(hgf, n):
    """A captured forward writes the integer accumulators where hgf_group_debug last said, also when that was after the
    capture - one launch and two."""
    M, K, N, r = 2, 512, 72, 16
    problems = []
    for i in range(n):
        x, packed, gamma, c = layer(hgf, M, K, N, r, i)
        problems.append({"x": x, "d_in": K, "d_out": N, "packed": packed, "gamma": gamma, "y": torch.empty((M, N), device="cuda"), **c})
    group = hgf.Group(problems)
    before = hgf.launch_count()
    group.forward()
    assert hgf.launch_count() - before == (1 if n == 3 else 2)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        group.forward()
    y_int = torch.full((M, N), -7, dtype=torch.int32, device="cuda")
    xq = group.debug(1, y_int)["xq"]
    graph.replay()
    torch.cuda.synchronize()
    T = hgf.unpack_ternary(problems[1]["packed"], N, K)
    assert torch.equal(y_int.double(), xq.double() @ T.double().T)
    group.debug(1, None)
    y_int.fill_(-7)
    graph.replay()
    torch.cuda.synchronize()
    assert bool((y_int == -7).all())
    hgf.check_status()
    del graph
    group.close()


# One CTA an SM: two token tiles with more row tiles than run at once, more shared memory than lets two share an SM - in one round
# and, where the larger shares don't fit, in two.
ONE_ROUND = [[(16, 512, 5632, 32)], [(12, 64, 4096, 0)], [(9, 640, 3000, 64)] * 2, [(4, 2048, 2048, 64)] * 4, [(2, 1024, 2816, 16)] * 5, [(1, 4096, 1536, 32)] * 8]


@pytest.mark.parametrize("shapes", ONE_ROUND)
def test_one_cta_an_sm(hgf, shapes):
    """A group against its two phases run apart: int32 accumulators bit for bit, y to 2e-5."""
    problems = []
    for i, (M, K, N, r) in enumerate(shapes):
        x, packed, gamma, c = layer(hgf, M, K, N, r, 17 * i + K)
        problems.append({"x": x, "d_in": K, "d_out": N, "packed": packed, "gamma": gamma, "y": torch.empty((M, N), device="cuda"), **c})
    group = hgf.Group(problems)
    yi = [torch.empty(p["y"].shape, dtype=torch.int32, device="cuda") for p in problems]
    for i, t in enumerate(yi):
        group.debug(i, t)
    before = hgf.launch_count()
    group.forward()
    assert hgf.launch_count() - before == 1
    hgf.check_status()
    y1, yi1 = [p["y"].clone() for p in problems], [t.clone() for t in yi]
    for p, t in zip(problems, yi):
        p["y"].fill_(float("nan"))
        t.fill_(-1)
    group.forward_phases(1)
    group.forward_phases(2)
    hgf.check_status()
    for p, t, a, b in zip(problems, yi, y1, yi1):
        assert torch.equal(t, b)
        assert float((p["y"] - a).abs().max()) <= 2e-5 * float(a.abs().max())
    group.close()


# In the first two groups one problem asks for two token tiles: in the others the second tile has no token and reads the row of zeros.
UNEQUAL = [[(12, 320, 200, 32), (3, 640, 56, 16), (8, 512, 1000, 64), (1, 64, 24, 0)], [(9, 192, 72, 48), (16, 512, 512, 16), (1, 256, 17, 32)],
           [(5, 1024, 100, 16), (1, 1088, 300, 32), (7, 64, 2048, 64), (2, 704, 8, 0), (3, 320, 640, 48)]]


@pytest.mark.parametrize("shapes", UNEQUAL)
def test_group_of_unequal_problems(hgf, shapes):
    """Problems of unequal token counts, lengths and ranks in one launch, against the oracle: codes, scales and int32
    accumulators bit for bit, y to the decode path's 2e-5."""
    problems = []
    for i, (M, K, N, r) in enumerate(shapes):
        x, packed, gamma, c = layer(hgf, M, K, N, r, 31 * i + K)
        problems.append({"x": x, "d_in": K, "d_out": N, "packed": packed, "gamma": gamma, "y": torch.empty((M, N), device="cuda"), **c})
    group = hgf.Group(problems)
    yi = [torch.full((p["x"].shape[0], p["d_out"]), -1, dtype=torch.int32, device="cuda") for p in problems]
    views = [group.debug(i, t) for i, t in enumerate(yi)]
    before = hgf.launch_count()
    group.forward()
    assert hgf.launch_count() - before == 1
    hgf.check_status()
    whole = [p["y"].clone() for p in problems]
    for p, view, i in zip(problems, views, yi):
        T = hgf.unpack_ternary(p["packed"], p["d_out"], p["d_in"]).cpu().numpy()
        ref = oracle.forward(host(p["x"]), T, p["gamma"], host(p["At"]), host(p["Bt"]), host(p["gate"]))
        assert np.array_equal(host(view["xq"]), ref["xq"]) and np.array_equal(host(view["gamma_x"]), ref["gamma_x"])
        assert np.array_equal(host(i), ref["y_int"])
        assert np.abs(host(p["y"]) - ref["y"]).max() <= 2e-5 * np.abs(ref["y"]).max()
    # what the launch left in the workspace serves the group's contraction run on its own
    for p in problems:
        p["y"].fill_(float("nan"))
    group.forward_phases(2)
    hgf.check_status()
    for p, y in zip(problems, whole):
        assert float((p["y"] - y).abs().max()) <= 2e-5 * float(y.abs().max())
    group.close()
