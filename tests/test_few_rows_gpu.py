"""The path for few query rows (query heads of a KV group times query tokens: at most 24) at its edges, against the CPU
oracle: 1 row to 24 and the first size past it, key counts around the 128-key tile and around the sizes where the chunk of
a CTA grows, each producer, and a packed batch too large for the sequence table that travels with the launch."""
import numpy as np
import pytest
import torch

from paper_2609_09721_b200 import binding, inputs
from test_attention_gpu import MEAN, TOL_O, _all_rows, _case_tensors, _check_dump, _recorded

pytestmark = pytest.mark.gpu

# producer: (oracle path, tolerance)
PRODUCERS = {"efq": ("efq", TOL_O), "lut": ("efq_lut", TOL_O), "etq0": ("etq", 5e-3), "etq1": ("etq6", 5e-3), "etq2": ("etq", 5e-3),
             "etq3": ("etq", 5e-3), "etq4": ("etq_fp32den", 5e-3)}


def _forward(dq, dk, dv, causal, producer, threshold=0.0, debug=None):
    if producer.startswith("etq"):
        return binding.exp_then_quantize_attention_fwd(dq, dk, dv, causal, 0.0, int(producer[3:]), debug=debug)
    return binding.efq_attention_fwd(dq, dk, dv, causal, 0.0, (MEAN[0], MEAN[1], int(producer == "lut"), 0, threshold), debug=debug)


@pytest.mark.parametrize("Hq,Hkv,Sq,Sk,causal,producer,threshold", [
    (1, 1, 1, 1, True, "efq", 0.0), (4, 4, 1, 127, False, "efq", 0.0), (8, 1, 1, 129, True, "efq", 0.0),        # 1, 1, 8 rows
    (2, 2, 9, 2047, True, "efq", 0.0), (4, 1, 4, 2049, True, "efq", 0.0), (2, 1, 8, 128, False, "efq", 0.0),    # 9, 16, 16 rows
    (1, 1, 17, 4095, True, "efq", 0.0), (8, 1, 3, 4097, False, "efq", 0.0), (1, 1, 24, 16, True, "efq", 0.0),   # 17, 24, 24 rows
    (5, 1, 5, 1500, True, "efq", 0.0),                                                                        # 25 rows: the general path
    (8, 2, 1, 16385, True, "efq", 0.0), (6, 2, 2, 1793, True, "efq", 2.0),
    (2, 1, 4, 1, True, "lut", 0.0), (2, 1, 4, 1, True, "etq0", 0.0), (2, 1, 4, 1, True, "etq1", 0.0),           # three queries see nothing
    (2, 1, 4, 1, True, "etq2", 0.0), (2, 1, 4, 1, True, "etq3", 0.0), (2, 1, 4, 1, True, "etq4", 0.0), (1, 1, 8, 3, True, "etq0", 0.0),
    (2, 1, 8, 3968, True, "efq", 0.0), (2, 1, 8, 3969, True, "etq2", 0.0), (1, 1, 9, 600, True, "lut", 0.0),      # 16 rows: chunks of 2 and 8 tiles
    (8, 1, 3, 8064, False, "efq", 0.0), (1, 1, 17, 8065, True, "efq", 0.0), (8, 1, 3, 8193, False, "lut", 0.0),   # the line for 17 to 24 rows
    (3, 1, 7, 8300, True, "etq0", 0.0), (4, 1, 6, 9000, True, "etq1", 0.0), (1, 1, 24, 8192, True, "etq4", 0.0),
    (8, 2, 1, 1025, True, "lut", 0.0), (3, 1, 7, 600, True, "etq0", 0.0), (8, 2, 1, 2100, False, "etq1", 0.0), (4, 1, 6, 333, True, "etq2", 0.0),
])
def test_few_rows_against_the_oracle(oracle, Hq, Hkv, Sq, Sk, causal, producer, threshold):
    case = inputs.AttentionCase("few", 1, Hq, Hkv, Sq, Sk, 128, causal, 500 + Sk, "k_outliers")
    (q, k, v), (dq, dk, dv) = _case_tensors(case)
    head = Hq - 1
    dump = binding.DebugDump(0, head, 0, Sq, Sk)
    o = _forward(dq, dk, dv, causal, producer, threshold, debug=dump)
    production = _forward(dq, dk, dv, causal, producer, threshold)
    torch.cuda.synchronize()
    assert torch.equal(o, production)
    path, tol = PRODUCERS[producer]
    rows = np.array([(0, h, i) for h in range(Hq) for i in range(Sq)], np.int64)
    want = oracle.attention_rows(q, k, v, rows, causal, case.softmax_scale, path, rescale_threshold=threshold)
    got = o.cpu().numpy().reshape(-1, 128)
    assert np.abs(got - want).max() <= tol
    if causal and Sq > Sk:                      # queries before the first key see nothing
        assert np.all(got.reshape(Hq, Sq, 128)[:, : Sq - Sk] == 0.0)
    else:
        _check_dump(oracle, case, dump, _all_rows(case, head, 0, Sq), MEAN, producer=path.replace("_fp32den", ""), threshold=threshold)


@pytest.mark.parametrize("n_seqs,tokens", [(128, 12), (129, 12), (128, 4), (129, 4)])
def test_packed_batch_of_few_row_sequences(n_seqs, tokens):
    """128 sequences of few rows (4 tokens: up to 8) are described in the launch itself, more in device memory; of those with up to
    12 tokens some go the general way beside them.  Each equals its forward alone bit for bit."""
    Hq, Hkv = 4, 2
    g = torch.Generator(device="cuda").manual_seed(7)
    lens = [(1 + n % tokens, 1 + (37 * n) % 700) for n in range(n_seqs)]
    cu_q = np.concatenate([[0], np.cumsum([a for a, _ in lens])])
    cu_k = np.concatenate([[0], np.cumsum([b for _, b in lens])])
    q = torch.randn(int(cu_q[-1]), Hq, 128, generator=g, device="cuda").bfloat16()
    k, v = (torch.randn(int(cu_k[-1]), Hkv, 128, generator=g, device="cuda").bfloat16() for _ in range(2))
    o = binding.efq_attention_fwd_varlen(q, k, v, cu_q, cu_k, True)
    for n in range(n_seqs):
        a, b, c, d = cu_q[n], cu_q[n + 1], cu_k[n], cu_k[n + 1]
        alone = binding.efq_attention_fwd(*(t.permute(1, 0, 2)[None].contiguous() for t in (q[a:b], k[c:d], v[c:d])), True)
        assert torch.equal(o[a:b].permute(1, 0, 2), alone[0]), f"sequence {n}"


@pytest.mark.parametrize("Hq,Hkv,Sq,Sk,B,producer,threshold", [
    (4, 4, 1, 2049, 8, "efq", 0.0), (4, 4, 1, 3968, 8, "etq4", 0.0),      # chunks of 2 tiles, the last of 1; 31 tiles
    (32, 8, 1, 8191, 4, "efq", 0.0), (8, 1, 1, 8300, 30, "lut", 0.0),     # 4 tiles, 16 chunks; 17, the last of 1 tile
    (2, 2, 1, 20000, 12, "efq", 0.0), (1, 1, 1, 16385, 20, "etq0", 0.0),  # 8 tiles; the last chunk of 5 and of 1
    (1, 1, 9, 4097, 80, "efq", 0.0), (16, 2, 2, 4200, 30, "efq", 1.0),    # 9 and 16 rows: chunks of 8 from 32 tiles on
    (8, 1, 3, 8193, 40, "efq", 0.0), (8, 2, 5, 9000, 20, "etq2", 0.0),    # 24 and 20 rows
    (288, 18, 1, 1000, 4, "efq", 0.0), (296, 37, 1, 2100, 4, "efq", 0.0),   # 288 rows: in parts by itself; 296, but too many chunks
    (304, 19, 1, 1000, 4, "efq", 0.0), (512, 32, 1, 4200, 2, "efq", 0.0),  # more rows than that: whole; in parts with chunks of 8
])
def test_chunks_in_parts_equal_whole_chunks(Hq, Hkv, Sq, Sk, B, producer, threshold):
    """Where few chunks do not fill the chip they are taken in parts, tile by tile: a sequence by itself gives the bits that it
    gives in a batch of B, whose chunks (more than 222) are taken whole."""
    g = torch.Generator(device="cuda").manual_seed(Sk)
    q = torch.randn(B, Hq, Sq, 128, generator=g, device="cuda").bfloat16()
    k, v = (torch.randn(B, Hkv, Sk, 128, generator=g, device="cuda").bfloat16() for _ in range(2))
    batch = _forward(q, k, v, True, producer, threshold)
    for b in (0, B - 1):
        assert torch.equal(_forward(q[b:b + 1].contiguous(), k[b:b + 1].contiguous(), v[b:b + 1].contiguous(), True, producer, threshold)[0], batch[b])


@pytest.mark.parametrize("Hq,Hkv,Sq,Sk,parts", [
    (288, 18, 1, 1000, True), (304, 19, 1, 1000, False),                   # chunks of two: as many rows as the merge takes at once, more
    (512, 32, 1, 4200, True), (1024, 64, 1, 600, False), (32, 8, 1, 8191, True), (8, 2, 1, 5000, True), (8, 8, 1, 500, False),
])
def test_where_chunks_are_taken_in_parts(Hq, Hkv, Sq, Sk, parts):
    g = torch.Generator(device="cuda").manual_seed(1)
    q = torch.randn(1, Hq, Sq, 128, generator=g, device="cuda").bfloat16()
    k, v = (torch.randn(1, Hkv, Sk, 128, generator=g, device="cuda").bfloat16() for _ in range(2))
    assert any("few_merge_tiles_kernel" in name for name, _ in _recorded(lambda: binding.efq_attention_fwd(q, k, v, True))) == parts


@pytest.mark.parametrize("seqs,Hq,Hkv,producer", [
    ([(1, 700), (1, 2100), (1, 5000), (1, 20000)], 8, 1, 0),               # 1, 2, 4 and 8 tiles a chunk in one launch
    ([(1, 700), (2, 9000), (3, 8300), (1, 130), (2, 4100)], 8, 1, 0),      # of 8, 16 and 24 rows
    ([(1, 20000), (4, 3000), (1, 1), (2, 2100)], 8, 2, 4), ([(1, 5000), (1, 300), (1, 16500)], 4, 2, 1),
])
def test_packed_sequences_in_parts(seqs, Hq, Hkv, producer):
    """A packed batch of few contexts is taken tile by tile, whatever the lengths of their chunks and their rows: each sequence gives
    the bits of its forward in a dense batch large enough to be taken in whole chunks."""
    g = torch.Generator(device="cuda").manual_seed(11)
    cu_q = np.concatenate([[0], np.cumsum([a for a, _ in seqs])])
    cu_k = np.concatenate([[0], np.cumsum([b for _, b in seqs])])
    q = torch.randn(int(cu_q[-1]), Hq, 128, generator=g, device="cuda").bfloat16()
    k, v = (torch.randn(int(cu_k[-1]), Hkv, 128, generator=g, device="cuda").bfloat16() for _ in range(2))
    call = lambda: binding.efq_attention_fwd_varlen(q, k, v, cu_q, cu_k, True, 0.0, producer)
    assert any("few_merge_tiles_kernel" in kernel for kernel, _ in _recorded(call))
    o = call()
    name = {0: "efq", 1: "etq0", 4: "etq2"}[producer]
    for n, (lq, lk) in enumerate(seqs):
        a, b, c, d = cu_q[n], cu_q[n + 1], cu_k[n], cu_k[n + 1]
        copies = 300 if lk < 8192 else 160                     # more than 222 chunks
        dense = [t.permute(1, 0, 2)[None].expand(copies, -1, -1, -1).contiguous() for t in (q[a:b], k[c:d], v[c:d])]
        assert torch.equal(o[a:b].permute(1, 0, 2), _forward(*dense, True, name)[copies - 1]), f"sequence {n}"


@pytest.mark.parametrize("Hq,Hkv,Sq,Sk", [
    (8, 8, 1, 500), (32, 8, 1, 1000), (1, 1, 1, 1000), (1, 1, 1, 60),        # chunks of one tile
    (4, 4, 1, 3000), (16, 1, 1, 1000), (16, 4, 4, 1500), (1, 1, 16, 100),    # of two; one tile in a chunk of two
    (32, 8, 1, 8191), (2, 2, 1, 16384), (1, 1, 16, 4096), (1, 1, 24, 8192),  # of four, eight
])
def test_no_block_without_a_tile(Hq, Hkv, Sq, Sk):
    """A chunk is cut into as many blocks as it has tiles at most: the streaming kernels launch no more blocks than there are tiles."""
    g = torch.Generator(device="cuda").manual_seed(1)
    q = torch.randn(1, Hq, Sq, 128, generator=g, device="cuda").bfloat16()
    k, v = (torch.randn(1, Hkv, Sk, 128, generator=g, device="cuda").bfloat16() for _ in range(2))
    launched = _recorded(lambda: binding.efq_attention_fwd(q, k, v, True))
    blocks = {n: grid for name, grid in launched for n in ("few_scores", "few_values") if n in name}
    assert sorted(blocks) == ["few_scores", "few_values"]
    assert max(blocks.values()) <= Hkv * ((Sk + 127) // 128)


@pytest.mark.parametrize("S,Hq,Hkv", [(127, 2, 1), (129, 1, 1), (257, 3, 3)])
def test_inputs_at_a_16_byte_boundary(S, Hq, Hkv):
    """Operand preparation loads 32 bytes at a time where the input allows it: inputs that start 16 bytes off give the same."""
    g = torch.Generator(device="cuda").manual_seed(11)

    def pair(heads):
        t = torch.randn(1, heads, S, 128, generator=g, device="cuda").bfloat16()
        shifted = torch.empty(t.numel() + 16, dtype=torch.bfloat16, device="cuda")[8:8 + t.numel()].view(t.shape)
        return t, shifted.copy_(t)

    (q, q2), (k, k2), (v, v2) = pair(Hq), pair(Hkv), pair(Hkv)
    assert torch.equal(binding.efq_attention_fwd(q, k, v, True), binding.efq_attention_fwd(q2, k2, v2, True))


@pytest.mark.parametrize("B,Hq,Hkv,Sq,Sk", [(1, 4, 4, 1, 700), (1, 8, 2, 3, 1500), (2, 2, 2, 24, 8100)])
@pytest.mark.parametrize("value", [float("inf"), float("-inf"), float("nan"), 3.38e38])
@pytest.mark.parametrize("where", ["q", "k", "v"])
def test_non_finite_inputs_as_on_the_general_path(B, Hq, Hkv, Sq, Sk, value, where):
    """Infinities, NaN and the largest values (whose scores overflow): the row maximum is infinite from some tile on, and the
    chunks add up as on the general path, which the two-call form always takes.  Both add FP32 numbers in different orders:
    2^-23 per addition of a tile, below 1e-5 of the row's largest value."""
    g = torch.Generator(device="cuda").manual_seed(Sk)
    t = {"q": torch.randn(B, Hq, Sq, 128, generator=g, device="cuda").bfloat16(),
         "k": torch.randn(B, Hkv, Sk, 128, generator=g, device="cuda").bfloat16(),
         "v": torch.randn(B, Hkv, Sk, 128, generator=g, device="cuda").bfloat16()}
    x = t[where].view(-1)
    if where == "v":
        value = min(max(value, -1e30), 1e30) if value == value else 1e30     # larger ones overflow in one order of the sum and not in another
    x[torch.randint(0, x.numel(), (max(1, x.numel() // 2000),), generator=g, device="cuda")] = value
    q, k, v = t["q"], t["k"], t["v"]
    shape = (B, Hq, Hkv, Sq, Sk, 128)
    ws = torch.empty(binding.efq_attention_workspace_bytes(*shape), dtype=torch.uint8, device="cuda")
    for causal in (False, True):
        for producer in (0, 1, 4):
            got = binding.exp_then_quantize_attention_fwd(q, k, v, causal, 0.0, {1: 0, 4: 2}[producer]) if producer else binding.efq_attention_fwd(q, k, v, causal)
            binding.efq_quantize_qkv(q, k, v, ws)
            want = binding.efq_attention_fwd_quantized(torch.empty_like(got), shape, ws, causal, 0.0, producer)
            assert torch.isfinite(want).all()
            scale = want.abs().amax(dim=-1, keepdim=True)
            assert ((got - want).abs() <= 1e-5 * scale).all(), (causal, producer)


def test_rows_past_two_to_the_31_scores():
    """24 rows on 98 million keys: the scores of rows 22 and 23 start past 2^31.  Every row asks the same, so every row answers
    what one row by itself does, bit for bit (both lengths of context are cut into the same chunks)."""
    Sk = 98_000_001
    assert 22 * Sk > 2 ** 31
    g = torch.Generator(device="cuda").manual_seed(17)
    kv = torch.empty(1, 1, Sk, 128, dtype=torch.bfloat16, device="cuda").normal_(generator=g)
    q = torch.randn(1, 1, 1, 128, generator=g, device="cuda").bfloat16()
    one = binding.efq_attention_fwd(q, kv, kv)
    rows = binding.efq_attention_fwd(q.expand(1, 1, 24, 128).contiguous(), kv, kv)
    assert torch.isfinite(one).all() and one.abs().max() > 0
    for r in range(24):
        assert torch.equal(rows[0, 0, r], one[0, 0, 0]), f"row {r}"
    del kv, one, rows
    torch.cuda.empty_cache()
