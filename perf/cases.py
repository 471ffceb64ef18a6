"""Timed cases of the library: what a program that serves a model with it calls, through the public binding.

`listed()` is a fixed set, `draw(rng)` gives one more case of the same ranges, `prepare(case, seed)` makes what the
program has in hand before the call (weights, activations, output buffers, the plan), `run(state)` is one pass.
Every result is compared bit for bit: a shape defines its reduction order, so any correct build gives the same bits.

The kinds of work:
  linear   one linear layer on device activations (decode M <= 64, prefill above), weights in BF16, FP16 or FP32
  norm     RMSNorm followed by the projection that reads it (the entry of an attention or feed-forward block)
  head     the LM head and the greedy token of every row
  attn     decode attention over a key/value cache with grouped-query heads
  host     one linear layer whose activations arrive in pinned host memory and whose result goes back there
  noalloc  one linear layer in a program that may not allocate (no plan)
"""
import math

import torch

from paper_2609_25624_b200 import binding as B
from paper_2609_25624_b200 import inputs

# (K, N) of the projections of a Llama-3-8B-architecture layer
LAYER = [(K, N) for (_, K, N) in inputs.LLAMA3_8B_LAYER]
HEAD_K, HEAD_N = inputs.LLAMA3_8B_LM_HEAD[1:]
WEIGHT_BYTES = {"bf16": 2, "fp16": 2, "fp32": 4}
EPS = 1e-5


def _linear(name, M, N, K, w="bf16", bias=True, kind="linear"):
    return {"name": name, "kind": kind, "M": M, "N": N, "K": K, "w": w, "bias": bias}


def _attn(name, batch, T, D=128, Hq=32, Hkv=8):
    return {"name": name, "kind": "attn", "batch": batch, "T": T, "D": D, "Hq": Hq, "Hkv": Hkv}


def listed():
    return [
        # the smallest layer of the test configurations: one row, launch latency is everything
        _linear("tiny_m1", 1, 1024, 512),
        # entry of a decode step's attention block for four sequences: weights stream from memory
        _linear("norm_qkv_m4", 4, 6144, 4096, bias=False, kind="norm"),
        # the widest projection of a decode step at a middle batch, weights kept as FP16
        _linear("gate_up_m16_fp16", 16, 28672, 4096, w="fp16"),
        # the deepest projection at the largest measured decode batch
        _linear("down_m32", 32, 4096, 14336),
        # LM head and greedy token at batch 8
        _linear("lm_head_m8", 8, HEAD_N, HEAD_K, bias=False, kind="head"),
        # a layer whose K is no multiple of the vector width (feature counts as they come)
        _linear("ragged_m6", 6, 1333, 1001),
        # the 100 x 1000 x 1000 probe shape with FP32 weights: a small ragged prefill
        _linear("probe_m100_fp32", 100, 1000, 1000, w="fp32"),
        # prompt of 512 tokens through the widest projection
        _linear("prefill_gate_up_m512", 512, 28672, 4096),
        # prompt of 2048 tokens through the deepest projection: the largest call
        _linear("prefill_down_m2048", 2048, 4096, 14336),
        # one decode step's attention: eight sequences with 4096 cached keys, grouped-query heads
        _attn("attention_b8_t4096", 8, 4096),
        # activations from and to pinned host memory around one output projection
        _linear("host_o_m8", 8, 4096, 4096, kind="host"),
        # the same projection in a latency-critical loop that may not allocate
        _linear("noalloc_o_m3", 3, 4096, 4096, bias=False, kind="noalloc"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _layer_or_generic(rng, most_elements=28672 * 4096):
    """(K, N) of a model layer, or generic sizes: K a multiple of 8, N anything."""
    if rng.random() < 0.4:
        return rng.choice(LAYER)
    K = 8 * _log(rng, 32, 1792)
    return K, _log(rng, 256, max(257, min(28672, most_elements // K)))


def draw(rng):
    kind = rng.choice(["decode", "decode", "prefill", "prefill", "norm", "head", "ragged", "attn", "host", "noalloc"])
    if kind == "attn":
        T = _log(rng, 128, 8192)
        batch = _log(rng, 1, min(32, 131072 // T))
        return {k: v for k, v in _attn("", batch, T, rng.choice([64, 128, 128]), *rng.choice([(32, 8), (32, 8), (16, 2), (8, 8)])).items()
                if k != "name"}
    w, bias, sort = "bf16", rng.random() < 0.5, "linear"
    if kind == "decode":
        K, N = _layer_or_generic(rng)
        M, w = _log(rng, 1, 64), rng.choice(["bf16", "bf16", "fp16", "fp32"])
    elif kind == "prefill":
        K, N = _layer_or_generic(rng)
        most = int(2048 * 4096 * 14336 // (N * K))       # no more multiply-adds than the largest listed case
        M, w = _log(rng, 65, max(66, min(2048, most))), rng.choice(["bf16", "bf16", "fp16", "fp32"])
    elif kind == "norm":
        sort, bias = "norm", False
        K, N = 128 * _log(rng, 8, 64), _log(rng, 1024, 28672)
        M = _log(rng, 1, 64)
    elif kind == "head":
        sort, bias = "head", False
        K, N, M = 128 * _log(rng, 8, 32), _log(rng, 16384, HEAD_N), _log(rng, 1, 32)
    elif kind == "ragged":
        K, N, M = 2 * _log(rng, 50, 2048) + 1, _log(rng, 64, 8192), _log(rng, 1, 300)
        w = rng.choice(["bf16", "bf16", "fp32"])
    elif kind == "host":
        sort = "host"
        (K, N), M = _layer_or_generic(rng), _log(rng, 1, 64)
    else:
        sort = "noalloc"
        (K, N), M = _layer_or_generic(rng, 4096 * 14336), _log(rng, 1, 32)
        if N * K > 4096 * 14336:
            K, N = 4096, 4096
    return {"kind": sort, "M": M, "N": N, "K": K, "w": w, "bias": bias}


def prepare(case, seed):
    g = torch.Generator(device="cuda").manual_seed(int(seed))

    def normal(*shape):
        return torch.randn(*shape, dtype=torch.float32, device="cuda", generator=g)

    s = {"kind": case["kind"]}
    if case["kind"] == "attn":
        b, T, D, Hq, Hkv = (case[k] for k in ("batch", "T", "D", "Hq", "Hkv"))
        s.update(q=normal(b, Hq, D), k=normal(b, Hkv, T, D), v=normal(b, Hkv, T, D), scale=1.0 / math.sqrt(D),
                 o=torch.empty(b, Hq, D, dtype=torch.float32, device="cuda"))
        return s
    M, N, K = case["M"], case["N"], case["K"]
    s["W"] = (0.02 * normal(N, K)).to(inputs.WEIGHT_DTYPES[case["w"]])
    s["x"] = normal(M, K)
    s["b"] = 0.01 * normal(N) if case["bias"] else None
    s["y"] = torch.empty(M, N, dtype=torch.float32, device="cuda")
    if case["kind"] != "noalloc":
        s["plan"] = B.det_linear_plan(M, N, K) if case["w"] == "bf16" else B.det_linear_plan_w(M, N, K, case["w"])
    if case["kind"] == "norm":
        s["gain"] = 1.0 + 0.1 * normal(K)
        s["h"] = torch.empty(M, K, dtype=torch.float32, device="cuda")
    elif case["kind"] == "head":
        s["idx"] = torch.empty(M, dtype=torch.int32, device="cuda")
    elif case["kind"] == "host":
        s["x"] = s["x"].cpu().pin_memory()
        s["y"] = torch.empty(M, N, dtype=torch.float32).pin_memory()
    return s


def run(s):
    kind = s["kind"]
    if kind == "linear":
        B.det_linear_run(s["plan"], s["x"], s["W"], s["b"], s["y"])
        return s["y"]
    if kind == "norm":
        B.det_rmsnorm(s["x"], s["gain"], EPS, s["h"])
        B.det_linear_run(s["plan"], s["h"], s["W"], s["b"], s["y"])
        return s["h"], s["y"]
    if kind == "head":
        B.det_linear_run(s["plan"], s["x"], s["W"], s["b"], s["y"])
        B.det_argmax_rows(s["y"], s["idx"])
        return s["y"], s["idx"]
    if kind == "attn":
        B.det_attention_decode(s["q"], s["k"], s["v"], s["scale"], s["o"])
        return s["o"]
    if kind == "host":
        B.det_linear_run_host(s["plan"], s["x"], s["W"], s["b"], s["y"])
        return s["y"]
    B.det_linear_run_noalloc(s["x"], s["W"], s["b"], s["y"])
    return s["y"]


def work(case):
    """Inputs read once, outputs written once; multiply-adds counted as two operations."""
    if case["kind"] == "attn":
        b, T, D, Hq, Hkv = (case[k] for k in ("batch", "T", "D", "Hq", "Hkv"))
        return {"bytes": 4 * (2 * b * Hkv * T * D + 2 * b * Hq * D), "flops": 4 * b * Hq * T * D}
    M, N, K = case["M"], case["N"], case["K"]
    w = {"bytes": WEIGHT_BYTES[case["w"]] * N * K + 4 * M * K + 4 * M * N + (4 * N if case["bias"] else 0), "flops": 2 * M * N * K}
    if case["kind"] == "norm":
        w["bytes"] += 4 * M * K + 4 * K              # the normalised rows are an output, the gain an input
        w["flops"] += 4 * M * K
    elif case["kind"] == "head":
        w["bytes"] += 4 * M
    return w


def tolerance(case):
    """The order of every reduction is a function of the shape alone and each step is one IEEE operation."""
    return "exact"
