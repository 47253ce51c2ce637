"""Performance cases of the EFQ-Softmax attention library: the calls its users make, over their ranges.

Four kinds of call, all through paper_2609_09721_b200.binding:

  attention   one [B, H, S, 128] problem: efq_attention_fwd (affine rule or LUT variant) or, for the producers
              "etq0" .. "etq4", exp_then_quantize_attention_fwd with that scale mode
  varlen      a packed batch of sequences of mixed lengths: efq_attention_fwd_varlen
  stage       the probability-generation stage on a score matrix: efq_probgen, exp_then_quantize_probgen
  calibrate   what the calibration tool does for one workload: FP32 reference output, then the (tau, h) grid search

Shapes and value distributions are those of the package's own workloads (inputs.py): Qwen3-8B-shaped GQA prefill
with K outlier channels, WAN2.2-shaped non-causal attention with a smooth low-rank component, i.i.d. normal heads.
"""
import math
import random

import torch

from paper_2609_09721_b200 import binding

D = 128
POINTS = {"mean": (-3.06, 2.30), "mmlu": (-2.90, 2.00), "balance": (-2.10, 2.70)}   # the printed operating points
TAUS, HS = (-3.6, -3.06, -2.6, -2.1), (1.7, 2.0, 2.3, 2.7)


def _attention(name, Hq, Hkv, Sq, Sk, causal, recipe, producer="efq", B=1, point="mean"):
    c = {"kind": "attention", "producer": producer, "point": point, "B": B, "Hq": Hq, "Hkv": Hkv, "Sq": Sq, "Sk": Sk,
         "causal": causal, "recipe": recipe}
    return dict(c, name=name) if name else c


def _varlen(name, Hq, Hkv, n_seqs, q_min, q_max, k_min, k_max, self_attention, causal, lengths, producer="efq"):
    c = {"kind": "varlen", "producer": producer, "Hq": Hq, "Hkv": Hkv, "n_seqs": n_seqs, "q_min": q_min, "q_max": q_max,
         "k_min": k_min, "k_max": k_max, "self_attention": self_attention, "causal": causal, "lengths": lengths}
    return dict(c, name=name) if name else c


def _stage(name, rows, cols, pad, producer="efq"):
    c = {"kind": "stage", "producer": producer, "rows": rows, "cols": cols, "pad": pad}
    return dict(c, name=name) if name else c


def _calibrate(name, Hq, Hkv, S, causal, recipe, n_tau, n_h):
    c = {"kind": "calibrate", "Hq": Hq, "Hkv": Hkv, "S": S, "causal": causal, "recipe": recipe, "n_tau": n_tau, "n_h": n_h}
    return dict(c, name=name) if name else c


def listed():
    return [
        # one short head: the smallest call, all launch and pipeline latency
        _attention("single_head_1024", 1, 1, 1024, 1024, False, "iid"),
        # one decode step of one conversation: a single query token against a ragged context
        _attention("decode_one_8191", 32, 8, 1, 8191, True, "k_outliers"),
        # prompt processing: a short prompt, the benchmark's prompt, a very long document
        _attention("prefill_2048", 32, 8, 2048, 2048, True, "k_outliers"),
        _attention("prefill_16384", 32, 8, 16384, 16384, True, "k_outliers"),
        _attention("prefill_131072", 32, 8, 131072, 131072, True, "k_outliers"),
        # video diffusion: self-attention over a ragged token count, cross-attention to a text of 512 tokens
        _attention("video_self_32760", 24, 24, 32760, 32760, False, "lowrank"),
        _attention("video_cross_512", 24, 24, 32760, 512, False, "lowrank"),
        # the conventional MXFP4 path that the method is compared with, its default form
        _attention("exp_then_quantize_4096", 32, 8, 4096, 4096, True, "k_outliers", producer="etq0"),
        # serving: prompts of mixed lengths in one batch, a decode step over 64 conversations
        _varlen("serve_prefill_16", 32, 8, 16, 100, 3000, 0, 0, True, True, 1),
        _varlen("serve_decode_64", 32, 8, 64, 1, 1, 4096, 8192, False, True, 2),
        # the stage by itself on the stage configuration
        _stage("stage_4096x16384", 4096, 16384, 0),
        # the calibration tool on its default workload, a coarse grid
        _calibrate("calibrate_2048", 32, 8, 2048, True, "k_outliers", 4, 4),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


HEADS = [(1, 1), (4, 4), (8, 2), (16, 2), (24, 24), (28, 4), (32, 8), (32, 32)]
PAIRS_MAX = 32 * 131072.0 * 131072.0 / 2     # query-key pairs of the largest listed case


def draw(rng):
    """One more case of the same ranges."""
    while True:
        c = _draw(rng)
        if _pairs(c) <= 0.5 * PAIRS_MAX and work(c)["bytes"] <= 6e9:
            return c


def _draw(rng):
    kind = rng.choices(["prefill", "decode", "full", "cross", "varlen_prefill", "varlen_decode", "stage", "calibrate"],
                       [20, 12, 12, 10, 14, 14, 12, 6])[0]
    Hq, Hkv = rng.choice(HEADS)
    recipe = rng.choice(["iid", "k_outliers", "lowrank"])
    producer = rng.choices(["efq", "efq_lut", "etq0", "etq1", "etq2", "etq3", "etq4"], [12, 1, 1, 1, 1, 1, 1])[0]
    point = rng.choice(sorted(POINTS))
    B = rng.choice([1, 1, 1, 2, 3])
    if kind == "prefill":        # a prompt, now and then with tokens that are cached already
        S = _log(rng, 64, 100000)
        return _attention("", Hq, Hkv, S, S + rng.choice([0, 0, 0, rng.randint(1, 4000)]), True, recipe, producer, B, point)
    if kind == "decode":         # one token, or a few of a speculative step
        return _attention("", Hq, Hkv, rng.choice([1, 1, 1, 2, 5]), _log(rng, 100, 60000), True, recipe, producer, B, point)
    if kind == "full":
        S = _log(rng, 64, 60000)
        return _attention("", Hq, Hkv, S, S, False, recipe, producer, B, point)
    if kind == "cross":
        return _attention("", Hq, Hkv, _log(rng, 200, 60000), _log(rng, 30, 2000), False, recipe, producer, B, point)
    if kind == "varlen_prefill":
        top = _log(rng, 100, 8000)
        return _varlen("", Hq, Hkv, rng.randint(2, 40), max(1, top // 10), top, 0, 0, True, True, rng.randrange(1 << 20),
                       producer)
    if kind == "varlen_decode":
        top = _log(rng, 300, 20000)
        return _varlen("", Hq, Hkv, rng.randint(2, 128), 1, rng.choice([1, 1, 3]), max(1, top // 4), top, False, True,
                       rng.randrange(1 << 20), producer)
    if kind == "stage":
        return _stage("", _log(rng, 32, 16384), _log(rng, 100, 20000), rng.choice([0, 0, 4, 20]),
                      rng.choice(["efq", "efq", "efq", "efq_lut", "etq0", "etq2"]))
    return _calibrate("", Hq, Hkv, _log(rng, 200, 3000), rng.random() < 0.5, recipe, rng.randint(1, 4), rng.randint(1, 4))


def _lengths(case):
    """(query length, key length) of every sequence of a packed batch; a sequence of a step over cached tokens holds
    at least its own query tokens."""
    rng = random.Random(case["lengths"])
    out = []
    for _ in range(case["n_seqs"]):
        lq = rng.randint(case["q_min"], case["q_max"])
        out.append((lq, lq if case["self_attention"] else max(lq, rng.randint(case["k_min"], case["k_max"]))))
    return out


def _visible(lq, lk, causal):
    """Query-key pairs of one head."""
    if not causal:
        return lq * lk
    n = min(lq, lk)              # the last n queries see something
    return n * (lk - n) + n * (n + 1) // 2 if lk >= lq else n * (n + 1) // 2


def _pairs(case):
    if case["kind"] == "attention":
        return case["B"] * case["Hq"] * _visible(case["Sq"], case["Sk"], case["causal"])
    if case["kind"] == "varlen":
        return case["Hq"] * sum(_visible(lq, lk, case["causal"]) for lq, lk in _lengths(case))
    if case["kind"] == "calibrate":
        return case["Hq"] * _visible(case["S"], case["S"], case["causal"]) * (1 + case["n_tau"] * case["n_h"])
    return case["rows"] * case["cols"]


def work(case):
    if case["kind"] == "stage":
        rows, blocks = case["rows"], (case["cols"] + 31) // 32
        return {"bytes": rows * case["cols"] * 4 + rows * 4 + rows * blocks * 17, "flops": 6 * rows * case["cols"]}
    flops = 4 * D * _pairs(case)                       # the two contractions
    if case["kind"] == "varlen":
        tq = sum(lq for lq, _ in _lengths(case))
        tk = sum(lk for _, lk in _lengths(case))
        return {"bytes": (tq * case["Hq"] * 6 + tk * case["Hkv"] * 4) * D, "flops": flops}
    if case["kind"] == "calibrate":                    # operands once for the reference and once for the search, O_ref once
        return {"bytes": case["S"] * D * (case["Hq"] * 8 + case["Hkv"] * 8), "flops": flops}
    return {"bytes": case["B"] * D * (case["Hq"] * case["Sq"] * 6 + case["Hkv"] * case["Sk"] * 4), "flops": flops}


def tolerance(case):
    if case["kind"] == "stage":
        # integer decisions of an FP32 sequence that is part of the interface; the exponential producers differ where
        # the device's exponential sits on a rounding threshold
        return "exact" if case["producer"].startswith("efq") else {"rel": 0.0, "differ": 2e-3}
    if case.get("producer", "efq").startswith("etq"):
        return {"rel": 5e-3, "max": 0.5}               # E2M1 codes may flip where the exponential sits on a threshold
    return {"rel": 1e-5, "max": 2e-3}                  # FP32 sums in another order


def _normal(shape, gen, recipe, is_k):
    """bf16 [..., heads, tokens, 128] on the GPU."""
    x = torch.randn(shape, generator=gen, device="cuda", dtype=torch.bfloat16)
    heads, tokens = shape[-3], shape[-2]
    if recipe == "k_outliers" and is_k:                # 8 channels of every head ten times as large
        gain = torch.ones(shape[:-2] + (1, D), device="cuda", dtype=torch.bfloat16)
        channels = torch.rand(shape[:-2] + (1, D), generator=gen, device="cuda").argsort(-1)[..., :8]
        x.mul_(gain.scatter_(-1, channels, 10.0))
    elif recipe == "lowrank":                          # a smooth rank-16 component of RMS 2
        s = torch.arange(tokens, device="cuda", dtype=torch.float32)[:, None] / tokens
        freq = torch.arange(1, 17, device="cuda", dtype=torch.float32)
        for h in range(heads):
            phase = torch.rand(16, generator=gen, device="cuda")
            basis = torch.cos(2 * math.pi * (s * freq + phase)) * (2 * math.sqrt(2.0))
            x[..., h, :, :] += (basis @ (torch.randn(16, D, generator=gen, device="cuda") / 4)).to(torch.bfloat16)
    return x


def prepare(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    kind = case["kind"]
    if kind == "stage":
        rows, cols = case["rows"], case["cols"]
        ld = (cols + 3) // 4 * 4 + case["pad"]
        scores = torch.randn((rows, ld), generator=gen, device="cuda") * 3
        scores[torch.rand((rows, ld), generator=gen, device="cuda") < 0.01] = 12.0
        scores = scores[:, :cols]
        blocks = (cols + 31) // 32
        return {"case": case, "scores": scores, "row_max": scores.amax(1),
                "codes": torch.empty((rows, blocks * 16), dtype=torch.uint8, device="cuda"),
                "scales": torch.empty((rows, blocks), dtype=torch.uint8, device="cuda")}
    Hq, Hkv = case["Hq"], case["Hkv"]
    params = None
    if case.get("producer") == "efq_lut":
        params = binding.EfqParams(0.0, 1.0, 1, 0, 0.0)
    elif case.get("producer") == "efq":
        tau, h = POINTS[case.get("point", "mean")]
        params = binding.EfqParams(tau, h, 0, 0, 0.0)
    if kind == "varlen":
        lens = _lengths(case)
        cu_q, cu_k = [0], [0]
        for lq, lk in lens:
            cu_q.append(cu_q[-1] + lq)
            cu_k.append(cu_k[-1] + lk)
        q = torch.randn((cu_q[-1], Hq, D), generator=gen, device="cuda", dtype=torch.bfloat16)
        k = torch.randn((cu_k[-1], Hkv, D), generator=gen, device="cuda", dtype=torch.bfloat16)
        v = torch.randn((cu_k[-1], Hkv, D), generator=gen, device="cuda", dtype=torch.bfloat16)
        gain = torch.ones((1, Hkv, D), device="cuda", dtype=torch.bfloat16)
        channels = torch.rand((1, Hkv, D), generator=gen, device="cuda").argsort(-1)[..., :8]
        k.mul_(gain.scatter_(-1, channels, 10.0))
        n = case["n_seqs"]
        nbytes = binding.lib().efq_attention_varlen_workspace_bytes(
            (binding.C.c_int64 * (n + 1))(*cu_q), (binding.C.c_int64 * (n + 1))(*cu_k), n, Hq, Hkv, D)
        producer = {"efq": 0, "efq_lut": 0, "etq0": 1, "etq1": 2, "etq2": 4, "etq3": 5, "etq4": 6}[case["producer"]]
        return {"case": case, "q": q, "k": k, "v": v, "cu_q": cu_q, "cu_k": cu_k, "params": params, "producer": producer,
                "workspace": torch.empty(nbytes, dtype=torch.uint8, device="cuda")}
    B = case.get("B", 1)
    Sq, Sk = (case["S"], case["S"]) if kind == "calibrate" else (case["Sq"], case["Sk"])
    state = {"case": case, "params": params,
             "q": _normal((B, Hq, Sq, D), gen, case["recipe"], False),
             "k": _normal((B, Hkv, Sk, D), gen, case["recipe"], True),
             "v": _normal((B, Hkv, Sk, D), gen, case["recipe"], False),
             "o": torch.empty((B, Hq, Sq, D), dtype=torch.float32, device="cuda")}
    nbytes = binding.efq_attention_workspace_bytes(B, Hq, Hkv, Sq, Sk, D)
    state["workspace"] = torch.empty(nbytes, dtype=torch.uint8, device="cuda")
    return state


def run(state):
    case = state["case"]
    kind, producer = case["kind"], case.get("producer", "efq")
    if kind == "stage":
        if producer.startswith("etq"):
            return binding.exp_then_quantize_probgen(state["scores"], state["row_max"], 1.0, int(producer[3:]),
                                                     state["codes"], state["scales"])
        return binding.efq_probgen(state["scores"], state["row_max"], 1.0, (0.0, 1.0, 1) if producer == "efq_lut" else None,
                                   state["codes"], state["scales"])
    if kind == "varlen":
        return binding.efq_attention_fwd_varlen(state["q"], state["k"], state["v"], state["cu_q"], state["cu_k"],
                                                case["causal"], 0.0, state["producer"], state["params"], state["workspace"])
    if kind == "calibrate":
        o_ref = binding.efq_exact_attention_fwd(state["q"], state["k"], state["v"], case["causal"], 0.0, state["o"])
        rho, best = binding.efq_calibrate(state["q"], state["k"], state["v"], o_ref, TAUS[:case["n_tau"]], HS[:case["n_h"]],
                                          case["causal"], 0.0, state["workspace"])
        return {"o_ref": o_ref, "rho": rho, "best": best}
    if producer.startswith("etq"):
        return binding.exp_then_quantize_attention_fwd(state["q"], state["k"], state["v"], case["causal"], 0.0,
                                                       int(producer[3:]), state["o"], state["workspace"])
    return binding.efq_attention_fwd(state["q"], state["k"], state["v"], case["causal"], 0.0, state["params"], state["o"],
                                     state["workspace"])
