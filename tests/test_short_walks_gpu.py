"""Persistent CTAs (more query tiles than SMs), short KV walks and long ones: every row equals, bit for bit, what the kernel with one
CTA per query tile returns (it is the one that runs when the operand is dumped), and sampled rows match the CPU oracle.  Key
counts at the edges of a tile, ragged query tiles, GQA, batches, items without a visible key."""
import numpy as np
import pytest
import torch

from paper_2609_09721_b200 import binding, inputs
from test_attention_gpu import MEAN, TOL_O, _case_tensors, _recorded

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,Hq,Hkv,Sq,Sk,causal,producer,threshold", [
    (1, 24, 24, 1000, 1, False, "efq", 0.0), (1, 8, 2, 2500, 128, False, "efq", 0.0), (2, 8, 8, 1281, 129, False, "efq", 0.0),
    (1, 24, 24, 2100, 512, False, "efq", 0.0), (1, 12, 4, 3000, 1000, False, "efq", 0.0), (1, 8, 4, 2560, 5120, False, "efq", 0.0),
    (1, 8, 4, 2560, 5121, False, "efq", 0.0),                                # one key in the last tile
    (100, 4, 2, 127, 127, True, "efq", 0.0), (40, 4, 1, 130, 256, True, "efq", 0.0), (3, 16, 4, 600, 1024, True, "efq", 0.0),
    (5, 8, 2, 900, 200, True, "efq", 0.0),                                   # the first 700 queries see nothing
    (2, 16, 4, 700, 400, False, "efq", 1.0), (2, 16, 4, 700, 400, False, "lut", 0.0),
    (2, 16, 4, 700, 400, False, "etq0", 0.0), (2, 16, 4, 700, 400, False, "etq1", 0.0),
    (2, 16, 4, 700, 400, True, "etq2", 0.0), (2, 16, 4, 700, 400, False, "etq3", 0.0), (2, 16, 4, 700, 400, False, "etq4", 0.0),
    (1, 16, 4, 1300, 4000, True, "etq0", 0.0), (1, 16, 4, 1300, 4000, True, "etq2", 0.0), (2, 16, 4, 700, 400, True, "lut", 0.0), (1, 8, 2, 2600, 6400, True, "efq", 0.0),
    (1, 8, 4, 2560, 2048, False, "lut", 0.0), (1, 8, 4, 2560, 2049, False, "lut", 0.0),          # the other producers at the edge of a tile
    (1, 8, 4, 2560, 8192, False, "etq0", 0.0), (1, 8, 4, 2560, 8193, False, "etq1", 0.0), (1, 8, 4, 2560, 9000, False, "etq2", 0.0),
])
def test_short_walks_equal_one_cta_per_tile(oracle, B, Hq, Hkv, Sq, Sk, causal, producer, threshold):
    case = inputs.AttentionCase("short", B, Hq, Hkv, Sq, Sk, 128, causal, 600 + Sk, "k_outliers")
    (q, k, v), (dq, dk, dv) = _case_tensors(case)

    def forward(debug=None):
        if producer.startswith("etq"):
            return binding.exp_then_quantize_attention_fwd(dq, dk, dv, causal, 0.0, int(producer[3:]), debug=debug)
        return binding.efq_attention_fwd(dq, dk, dv, causal, 0.0, (MEAN[0], MEAN[1], int(producer == "lut"), 0, threshold), debug=debug)

    o = forward()
    assert torch.equal(o, forward(binding.DebugDump(B - 1, Hq - 1, 0, 1, Sk)))
    if producer in ("efq", "lut"):
        rng = np.random.default_rng(Sk)
        rows = np.stack([rng.integers(0, n, 64) for n in (B, Hq, Sq)], 1)
        rows[0], rows[1] = (0, 0, 0), (B - 1, Hq - 1, Sq - 1)
        want = oracle.attention_rows(q, k, v, rows, causal, case.softmax_scale, {"efq": "efq", "lut": "efq_lut"}[producer], rescale_threshold=threshold)
        got = o[rows[:, 0], rows[:, 1], rows[:, 2]].cpu().numpy()
        assert np.abs(got - want).max() <= TOL_O
    if causal and Sq > Sk:
        assert torch.all(o[:, :, : Sq - Sk] == 0)


@pytest.mark.parametrize("B,Hq,Hkv,Sq,Sk,producer", [
    (2, 16, 4, 1087, 470, "efq"), (8, 8, 8, 900, 200, "etq0"), (1, 32, 8, 2000, 1, "lut"),      # most items see nothing, and all but the last
    (20, 8, 8, 384, 128, "efq"), (20, 8, 8, 384, 129, "etq2"), (20, 8, 8, 384, 257, "efq"),      # whole tiles of zeros: two, one, one
])
def test_queries_before_the_first_key(B, Hq, Hkv, Sq, Sk, producer):
    """Causal with more queries than keys: the rows that see nothing are written as zeros, whole tiles of them by themselves; the others
    are those of the kernel with one CTA per query tile."""
    g = torch.Generator(device="cuda").manual_seed(Sq + Sk)
    q = torch.randn(B, Hq, Sq, 128, generator=g, device="cuda").bfloat16()
    k, v = (torch.randn(B, Hkv, Sk, 128, generator=g, device="cuda").bfloat16() for _ in range(2))

    def forward(debug=None):
        o = torch.full((B, Hq, Sq, 128), float("nan"), device="cuda")
        if producer.startswith("etq"):
            return binding.exp_then_quantize_attention_fwd(q, k, v, True, 0.0, int(producer[3:]), o, debug=debug)
        return binding.efq_attention_fwd(q, k, v, True, 0.0, (MEAN[0], MEAN[1], int(producer == "lut"), 0, 0.0), o, debug=debug)

    o = forward()
    assert torch.all(o[:, :, : Sq - Sk] == 0)
    assert torch.equal(o, forward(binding.DebugDump(0, Hq - 1, 0, 1, Sk)))


@pytest.mark.parametrize("Hq,Hkv,Sq,Sk,causal,producer,persistent", [
    (24, 24, 900, 30000, False, "efq", True), (32, 8, 20000, 20000, True, "efq", True),     # walks of 235 tiles, of 1 to 157
    (24, 24, 900, 6144, False, "lut", True), (24, 24, 900, 6145, False, "lut", False),      # the line of the table form, one key past it
    (24, 24, 900, 20000, False, "etq0", True), (24, 24, 900, 20000, False, "etq2", True), (24, 24, 900, 20000, False, "etq4", False),
    (1, 1, 148 * 128, 300, False, "efq", False), (1, 1, 148 * 128 + 1, 300, False, "efq", True),       # as many query tiles as SMs, one more
])
def test_long_walks_equal_one_cta_per_tile(Hq, Hkv, Sq, Sk, causal, producer, persistent):
    """Persistent CTAs in long walks, and which kernel runs at the lines of the rule: the bits of the kernel with one CTA per tile, which
    runs when the operand is dumped."""
    g = torch.Generator(device="cuda").manual_seed(Sk)
    q = torch.randn(1, Hq, Sq, 128, generator=g, device="cuda").bfloat16()
    k, v = (torch.randn(1, Hkv, Sk, 128, generator=g, device="cuda").bfloat16() for _ in range(2))

    def forward(debug=None):
        if producer.startswith("etq"):
            return binding.exp_then_quantize_attention_fwd(q, k, v, causal, 0.0, int(producer[3:]), debug=debug)
        return binding.efq_attention_fwd(q, k, v, causal, 0.0, (MEAN[0], MEAN[1], int(producer == "lut"), 0, 0.0), debug=debug)

    kernels = [name for name, _ in _recorded(forward)]
    assert any(("attention_short_kernel" if persistent else "attention_fwd_kernel") in name for name in kernels)
    assert torch.equal(forward(), forward(binding.DebugDump(0, Hq - 1, 0, 1, Sk)))


def test_a_forward_longer_than_the_limit_of_a_wait():
    """The limit (1.5e9 cycles, 0.76 s) is one on the time without another tile, not on that of a CTA: a forward of a second, all of it in
    the same CTAs, reports no problem, and its rows are those of short ones."""
    g = torch.Generator(device="cuda").manual_seed(9)
    q = torch.randn(1, 32, 340000, 128, generator=g, device="cuda", dtype=torch.bfloat16)
    k, v = (torch.randn(1, 1, 340000, 128, generator=g, device="cuda", dtype=torch.bfloat16) for _ in range(2))
    ws = torch.empty(binding.efq_attention_workspace_bytes(1, 32, 1, 340000, 340000, 128), dtype=torch.uint8, device="cuda")
    start, end = (torch.cuda.Event(enable_timing=True) for _ in range(2))
    o = torch.empty(1, 32, 340000, 128, device="cuda")
    start.record()
    binding.efq_attention_fwd(q, k, v, False, 0.0, None, o, ws)
    end.record()
    assert binding.efq_poll_status(ws) == 0
    assert start.elapsed_time(end) > 850.0
    for head, row in ((0, 0), (31, 339800)):
        few = q[:, head:head + 1, row:row + 200].contiguous()
        assert torch.equal(o[0, head, row:row + 200], binding.efq_attention_fwd(few, k, v)[0, 0])


@pytest.mark.parametrize("Hq,Hkv,causal,longest,producer", [(8, 2, True, 1000, 0), (6, 6, False, 5120, 0), (8, 4, True, 5121, 0), (8, 2, True, 700, 1), (8, 2, False, 512, 1)])
def test_short_walks_of_a_packed_batch(Hq, Hkv, causal, longest, producer):
    """Sequences of mixed lengths, whole last tiles and one key more: shared query tiles (few tokens), the
    few-row path beside them, queries that see nothing, none at all.  Each equals its forward alone bit for bit."""
    g = torch.Generator(device="cuda").manual_seed(13)
    lens = [(500, longest), (40, 300), (1, 200), (300, 100), (129, 129), (0, 50), (30, 257), (128, 128), (70, 0), (1300, min(640, longest)), (257, 384), (1000, 512)]
    cu_q = np.concatenate([[0], np.cumsum([a for a, _ in lens])])
    cu_k = np.concatenate([[0], np.cumsum([b for _, b in lens])])
    q = torch.randn(int(cu_q[-1]), Hq, 128, generator=g, device="cuda").bfloat16()
    k, v = (torch.randn(int(cu_k[-1]), Hkv, 128, generator=g, device="cuda").bfloat16() for _ in range(2))
    o = binding.efq_attention_fwd_varlen(q, k, v, cu_q, cu_k, causal, 0.0, producer)
    for n, (lq, lk) in enumerate(lens):
        got = o[cu_q[n]:cu_q[n + 1]].permute(1, 0, 2)
        if lq == 0 or lk == 0:
            assert torch.all(got == 0)
            continue
        one = [t.permute(1, 0, 2)[None].contiguous() for t in (q[cu_q[n]:cu_q[n + 1]], k[cu_k[n]:cu_k[n + 1]], v[cu_k[n]:cu_k[n + 1]])]
        alone = binding.exp_then_quantize_attention_fwd(*one, causal, 0.0, 0) if producer else binding.efq_attention_fwd(*one, causal)
        assert torch.equal(got, alone[0]), f"sequence {n}"


@pytest.mark.parametrize("Hq,Hkv,causal,producer,lens", [
    (8, 2, True, 0, [(20000, 20000), (300, 16000), (5000, 13000), (64, 64)]),         # walks of up to 157 tiles
    (4, 4, False, 1, [(1500, 13000), (13000, 1500), (400, 400)]), (8, 4, True, 4, [(14000, 14000), (3000, 9000), (129, 129)]),
    (2, 2, False, 0, [(3000, 3000)] + [(60 + 7 * n, 60 + 7 * n) for n in range(60)]),  # a few long ones among many short: not in turn
    (4, 4, True, 0, [(6000, 6000)] + [(50 + 7 * n, 50 + 7 * n) for n in range(63)]), (1, 1, True, 2, [(8000, 8000)] * 2 + [(80 + 12 * n, 80 + 12 * n) for n in range(60)]),
    (28, 4, False, 0, [(5000, 5000)] + [(1 + 5 * n, 1 + 5 * n) for n in range(60)]),   # shared query tiles and few rows beside them
    (2, 1, True, 0, [(9000, 9000), (4000, 300)] + [(90 + n, 10) for n in range(100)]),  # queries that see nothing, whole tiles of them
])
def test_long_walks_of_a_packed_batch(Hq, Hkv, causal, producer, lens):
    """Walks of a hundred and more KV tiles in a packed batch, and a few long sequences among many short ones, whose items do not go round
    in turn: each sequence equals its forward alone bit for bit."""
    g = torch.Generator(device="cuda").manual_seed(14)
    cu_q = np.concatenate([[0], np.cumsum([a for a, _ in lens])])
    cu_k = np.concatenate([[0], np.cumsum([b for _, b in lens])])
    q = torch.randn(int(cu_q[-1]), Hq, 128, generator=g, device="cuda").bfloat16()
    k, v = (torch.randn(int(cu_k[-1]), Hkv, 128, generator=g, device="cuda").bfloat16() for _ in range(2))
    o = binding.efq_attention_fwd_varlen(q, k, v, cu_q, cu_k, causal, 0.0, producer)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):                    # the table that the host wrote is read at every replay
        recorded = binding.efq_attention_fwd_varlen(q, k, v, cu_q, cu_k, causal, 0.0, producer)
    for _ in range(2):
        recorded.fill_(float("nan"))
        graph.replay()
        assert torch.equal(recorded, o)
    for n in range(len(lens)):
        one = [t.permute(1, 0, 2)[None].contiguous() for t in (q[cu_q[n]:cu_q[n + 1]], k[cu_k[n]:cu_k[n + 1]], v[cu_k[n]:cu_k[n + 1]])]
        alone = binding.exp_then_quantize_attention_fwd(*one, causal, 0.0, {1: 0, 2: 1, 4: 2}[producer]) if producer else binding.efq_attention_fwd(*one, causal)
        assert torch.equal(o[cu_q[n]:cu_q[n + 1]].permute(1, 0, 2), alone[0]), f"sequence {n}"
