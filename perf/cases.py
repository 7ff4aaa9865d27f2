"""What the performance of this framework is measured on: the calls a serving or evaluation program
makes, over the range of sizes it makes them at.

A case names a kind of call and its sizes:

  decode     a running batch goes on: `cycles` greedy (or sampled) decode cycles, and one cycle with
             given tokens, which hands out the logits of its passes
  prefill    a new batch of prompts: all prompt rows through all layers, the first token's logits and
             the KV cache
  score      logits of given sequences in one pass (the masked parallel forward)
  layer      one layer on new rows of every sequence against a filled KV cache
  attention  split-KV attention alone, on the caller's own cache

Shapes are the repository's: "qwen3_4b" is the 36-layer model the benchmark uses, "qwen3_4b_l4" its
4-layer stand-in where the prompt is too long to build 36 layers of cache quickly, "mid" and "tiny" the
small models of the tests.  Weights are random; the embedding is scaled up against the layers, so that
the model prefers one next token as clearly as a trained model does (the token just read): the tokens
of greedy cycles then do not hang on the last bits of the logits.
"""
import math

import torch

from paper_2510_11958_b200 import Dmtd, attention_decode, load_library
from synthetic import SHAPES, make_weights, weight_bytes

_KV_TYPES = {"f32": torch.float32, "bf16": torch.bfloat16, "f16": torch.float16}
_DECODE_ROOM = 2048            # positions a decode case may advance before the next request starts


def listed():
    return [
        # The smallest model of the tests, fp32 throughout: what a pass costs in launches and latency.
        {"name": "decode_tiny", "kind": "decode", "model": "tiny", "batch": 1, "prompt": 32, "L_d": 2, "tau": 3,
         "kv": "f32", "cycles": 7, "encoding_layers": 0, "temperature": 0.0},
        # One user of a chat: the benchmark's headline workload.
        {"name": "decode_b1", "kind": "decode", "model": "qwen3_4b", "batch": 1, "prompt": 512, "L_d": 8, "tau": 3,
         "kv": "f16", "cycles": 7, "encoding_layers": 0, "temperature": 0.0},
        # A few users, sampling: batches between the one-sequence and the many-sequence kernels.
        {"name": "decode_b3_sampled", "kind": "decode", "model": "qwen3_4b", "batch": 3, "prompt": 700, "L_d": 8, "tau": 3,
         "kv": "f16", "cycles": 5, "encoding_layers": 0, "temperature": 0.8},
        # A loaded server: the benchmark's batched workload.
        {"name": "decode_b32", "kind": "decode", "model": "qwen3_4b", "batch": 32, "prompt": 1024, "L_d": 8, "tau": 3,
         "kv": "f16", "cycles": 3, "encoding_layers": 0, "temperature": 0.0},
        # Long documents: decoding bound by the KV cache (bf16, as that workload has it).
        {"name": "decode_long_b8", "kind": "decode", "model": "qwen3_4b_l4", "batch": 8, "prompt": 16384, "L_d": 2, "tau": 3,
         "kv": "bf16", "cycles": 3, "encoding_layers": 0, "temperature": 0.0},
        # Time to the first token of one ordinary prompt.
        {"name": "prefill_b1", "kind": "prefill", "model": "qwen3_4b", "batch": 1, "prompt": 512, "kv": "f16"},
        # ... of one long document of no particular length: attention over thousands of positions.
        {"name": "prefill_long", "kind": "prefill", "model": "qwen3_4b_l4", "batch": 1, "prompt": 9001, "kv": "bf16"},
        # ... of the loaded server's whole batch, the largest call.
        {"name": "prefill_b32", "kind": "prefill", "model": "qwen3_4b", "batch": 32, "prompt": 1024, "kv": "f16"},
        # Evaluating two given answers: logits of every answer position.
        {"name": "score_b2", "kind": "score", "model": "qwen3_4b", "batch": 2, "prompt": 64, "tokens": 250, "L_d": 8, "tau": 3,
         "kv": "f16"},
        # A program that schedules layers itself (a cell of the single-layer grid).
        {"name": "layer_b64", "kind": "layer", "batch": 64, "rows": 1, "cached": 8192, "kv": "bf16"},
        # Attention inside someone else's decoder: one short sequence, and the refill rows of a long batch.
        {"name": "attention_b1", "kind": "attention", "batch": 1, "rows": 1, "keys": 1000, "q_heads": 32, "kv_heads": 8,
         "head_dim": 128, "kv": "f16"},
        {"name": "attention_b8_rows3", "kind": "attention", "batch": 8, "rows": 3, "keys": 16387, "q_heads": 32, "kv_heads": 8,
         "head_dim": 128, "kv": "bf16"},
    ]


def _spread(rng, lo, hi):
    """A whole number in [lo, hi], spread over its logarithm."""
    return min(hi, max(lo, round(math.exp(rng.uniform(math.log(lo), math.log(hi + 0.999)) - 0.25 / lo))))


def draw(rng):
    """One more case: the same kinds of call, sizes spread over the ranges the listed cases stand in."""
    kind = rng.choice(["decode", "decode", "decode", "prefill", "prefill", "score", "layer", "attention"])
    kv16 = rng.choice(["f16", "bf16"])
    if kind == "attention":
        head_dim, (q_heads, kv_heads) = rng.choice([(128, (32, 8)), (128, (8, 2)), (64, (16, 8))])
        kv = rng.choice([kv16, kv16, "f32"])
        batch = _spread(rng, 1, 64)
        rows = rng.choice([1, 1, 2, 3, 4])
        keys = _spread(rng, 16, 32768)
        keys = max(rows, min(keys, 524288 // batch))
        return {"kind": kind, "batch": batch, "rows": rows, "keys": keys, "q_heads": q_heads, "kv_heads": kv_heads,
                "head_dim": head_dim, "kv": kv}
    if kind == "layer":
        batch = _spread(rng, 1, 256)
        return {"kind": kind, "batch": batch, "rows": rng.choice([1, 1, 1, 2, 3, 4]),
                "cached": min(_spread(rng, 64, 32768), 1048576 // batch), "kv": kv16}
    model = rng.choice(["tiny", "mid", "qwen3_4b_l4", "qwen3_4b_l4", "qwen3_4b"])
    kv = "f32" if model == "tiny" else kv16
    layers = SHAPES[model].n_layers
    if kind == "prefill":
        batch = _spread(rng, 1, 32)
        most = {"tiny": 8192, "mid": 8192, "qwen3_4b_l4": 65536, "qwen3_4b": 16384}[model]
        return {"kind": kind, "model": model, "batch": batch, "prompt": min(_spread(rng, 5, 12000), most // batch), "kv": kv}
    L_d, tau = rng.choice([max(1, layers // 4), layers // 2]), rng.choice([1, 2, 3, 3, 3, 4])
    if kind == "score":
        batch = _spread(rng, 1, 4)
        prompt = _spread(rng, 1, 256)
        return {"kind": kind, "model": model, "batch": batch, "prompt": prompt, "tokens": prompt + _spread(rng, 4, 256),
                "L_d": L_d, "tau": tau, "kv": kv}
    batch = _spread(rng, 1, 32 if model == "qwen3_4b" else 64)
    most = {"tiny": 2048, "mid": 4096, "qwen3_4b_l4": 65536, "qwen3_4b": 16384}[model]
    return {"kind": kind, "model": model, "batch": batch, "prompt": min(_spread(rng, 8, 8192), most // batch), "L_d": L_d,
            "tau": tau, "kv": kv, "cycles": 3, "encoding_layers": rng.choice([0, 0, 0, 1]),
            "temperature": rng.choice([0.0, 0.0, 0.8])}


def _weights(shape, seed):
    """Random weights whose next token is clear (see above); norm weights around 1."""
    w = make_weights(shape, seed=seed, device="cuda", norm_jitter=0.1)
    w["embed"].mul_(128.0)
    w["final_norm"].mul_(1.0 / 64.0)
    return w


def _ids(shape, size, g):
    return torch.randint(0, shape.vocab, size, generator=g, dtype=torch.int32, device="cuda")


class _DeviceArray:
    """Device memory of a context as something torch can wrap without a copy; a tensor made of it keeps the
    context alive."""

    def __init__(self, eng, ptr, shape, typestr):
        self.eng = eng
        self.__cuda_array_interface__ = {"shape": tuple(shape), "typestr": typestr, "data": (int(ptr), False), "version": 2}


def _kv_views(eng, layer, kv):
    """K and V of one layer of a context: [max_batch, kv heads, max_seq, head_dim]."""
    s = eng.shape
    size = (eng.max_batch, s.n_kv_heads, eng.max_seq, s.head_dim)
    dtype = _KV_TYPES[kv]
    return [torch.as_tensor(_DeviceArray(eng, p, size, "<f4" if dtype == torch.float32 else "<i2"), device="cuda").view(dtype)
            for p in eng.kv(layer)]


def prepare(case, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    kind = case["kind"]
    if kind == "attention":
        B, R, n, nq, nkv, D = (case[k] for k in ("batch", "rows", "keys", "q_heads", "kv_heads", "head_dim"))
        cache = [torch.empty(B, nkv, n, D, dtype=_KV_TYPES[case["kv"]], device="cuda") for _ in range(2)]
        for t in cache:
            for b in range(B):
                t[b] = torch.randn(nkv, n, D, generator=g, device="cuda")
        need = load_library().dmtd_attention_scratch_bytes(B, R, nq, D, n)
        return {"kind": kind, "q": torch.randn(B, R, nq, D, generator=g, device="cuda"), "k": cache[0], "v": cache[1],
                "pos0": n - R, "scratch": torch.empty(max(need, 256), dtype=torch.uint8, device="cuda")}
    if kind == "layer":
        shape = SHAPES["qwen3_4b"].with_(n_layers=1, vocab=1024)
        B, R, n = case["batch"], case["rows"], case["cached"]
        eng = Dmtd(shape, make_weights(shape, seed=seed, device="cuda", norm_jitter=0.1), L_d=1, tau=1, max_batch=B,
                   max_seq=n + R, kv_dtype=case["kv"])
        for t in _kv_views(eng, 0, case["kv"]):
            for b in range(B):
                t[b, :, :n] = torch.randn(shape.n_kv_heads, n, shape.head_dim, generator=g, device="cuda")
        return {"kind": kind, "eng": eng, "hidden": torch.randn(B, R, shape.hidden, generator=g, device="cuda"),
                "work": torch.empty(B, R, shape.hidden, device="cuda"), "pos0": n}
    shape = SHAPES[case["model"]]
    B, P = case["batch"], case["prompt"]
    weights = _weights(shape, seed)
    if kind == "prefill":
        eng = Dmtd(shape, weights, L_d=max(1, shape.n_layers // 4), tau=3, max_batch=B, max_seq=P + 64, kv_dtype=case["kv"])
        cache = [t[:, :, :P] for t in _kv_views(eng, shape.n_layers - 1, case["kv"])]
        return {"kind": kind, "eng": eng, "prompt": _ids(shape, (B, P), g), "cache": cache}
    if kind == "score":
        eng = Dmtd(shape, weights, L_d=case["L_d"], tau=case["tau"], max_batch=B, max_seq=case["tokens"] + 64, kv_dtype=case["kv"])
        return {"kind": kind, "eng": eng, "tokens": _ids(shape, (B, case["tokens"]), g), "prompt_len": P}
    eng = Dmtd(shape, weights, L_d=case["L_d"], tau=case["tau"], max_batch=B, max_seq=P + _DECODE_ROOM, kv_dtype=case["kv"])
    if case["encoding_layers"]:
        eng.set_option("encoding_layers", case["encoding_layers"])
    if case["temperature"]:
        eng.set_sampling(case["temperature"], seed)
    state = {"kind": kind, "eng": eng, "prompt": _ids(shape, (B, P), g), "tau": case["tau"], "cycles": case["cycles"],
             "forced": _ids(shape, (B, case["tau"]), g)}
    _start_request(state)
    return state


def _start_request(state):
    """Prefill, and the rest of the cycle that it begins."""
    eng = state["eng"]
    eng.reset()
    eng.prefill(state["prompt"])
    while eng.state()["slot"] != 0:
        eng.decode_cycle(state["tau"])


def run(state):
    kind = state["kind"]
    if kind == "attention":
        return attention_decode(state["q"], state["k"], state["v"], state["pos0"], scratch=state["scratch"])
    eng = state["eng"]
    if kind == "layer":
        state["work"].copy_(state["hidden"])
        return eng.step_layers(0, 1, state["work"], state["pos0"])
    if kind == "prefill":
        eng.reset()
        _, logits = eng.prefill(state["prompt"], want_logits=True)
        return [logits] + state["cache"]
    if kind == "score":
        return eng.masked_forward(state["tokens"], state["prompt_len"])
    tau = state["tau"]
    if eng.state()["n_known"] + (state["cycles"] + 1) * tau > eng.max_seq:
        _start_request(state)                  # the cache is full: the next request
    tokens = [eng.decode_cycle(tau)[2] for _ in range(state["cycles"])]
    logits, _ = eng.decode_forced(state["forced"])
    return tokens, logits


def work(case):
    kind = case["kind"]
    kv_bytes = 4 if case["kv"] == "f32" else 2
    if kind == "attention":
        B, R, n, nq, nkv, D = (case[k] for k in ("batch", "rows", "keys", "q_heads", "kv_heads", "head_dim"))
        return {"bytes": 2 * B * nkv * n * D * kv_bytes + 2 * B * R * nq * D * 4, "flops": 4 * B * R * n * nq * D}
    if kind == "layer":
        shape = SHAPES["qwen3_4b"]
        rows, n = case["batch"] * case["rows"], case["cached"]
        w_layer, _ = weight_bytes(shape)
        return {"bytes": w_layer + 2 * case["batch"] * n * shape.kv_dim * kv_bytes + 2 * rows * shape.hidden * 4,
                "flops": 2 * rows * shape.params_per_layer + 4 * rows * n * shape.q_dim}
    shape = SHAPES[case["model"]]
    w_layer, w_head = weight_bytes(shape)
    B, P, L, head = case["batch"], case["prompt"], shape.n_layers, shape.vocab * shape.hidden
    per_pos = 2 * shape.kv_dim * kv_bytes
    if kind in ("prefill", "score"):
        n = P if kind == "prefill" else case["tokens"]
        out = 1 if kind == "prefill" else n - (P - 1)
        return {"bytes": L * w_layer + w_head + L * B * n * per_pos + B * out * shape.vocab * 4,
                "flops": B * n * L * (2 * shape.params_per_layer + 2 * n * shape.q_dim) + 2 * B * out * head}
    tau, n_cycles = case["tau"], case["cycles"] + 1
    short = case["L_d"] + case["encoding_layers"]
    passes = L + (tau - 1) * short                         # layers traversed in a cycle
    rows = B * ((L - short) * tau + tau * short)           # rows times layers
    cycle_bytes = passes * (w_layer + B * P * per_pos) + tau * w_head
    return {"bytes": n_cycles * cycle_bytes + tau * B * shape.vocab * 4,
            "flops": n_cycles * (rows * (2 * shape.params_per_layer + 4 * P * shape.q_dim) + 2 * B * tau * head)}


def tolerance(case):
    """Four times what was measured between this path and the same call with an fp32 cache (16-bit caches round
    K, V, the query and the probabilities once; fp16 has three bits more than bf16), with the largest differences
    of single values beside the norms; the order of the fp32 sums alone moves less than half as much."""
    kind, kv = case["kind"], case["kv"]
    differ = {"differ": 0.002} if kind == "decode" else {}
    if kv == "f32":
        return {"rel": 1e-5, "max": 1e-4, **differ}
    if kind == "attention":                    # against fp64: 2.4e-4 and 2.2e-3
        return {"rel": 1e-3, "max": 4e-3} if kv == "f16" else {"rel": 9e-3, "max": 5.4e-2}
    if kind == "prefill":                      # the cache rows themselves: 2.9e-4 and 1.7e-3
        return {"rel": 1.2e-3, "max": 1e-2} if kv == "f16" else {"rel": 7e-3, "max": 3.2e-2}
    if kind == "layer":                        # 1.0e-4 (bf16)
        return {"rel": 4e-4, "max": 2e-3}
    # logits: 0.9e-4 to 1.6e-4 over 36 layers with fp16; bf16 has eight times that rounding
    return {"rel": 6.5e-4, "max": 5.5e-3, **differ} if kv == "f16" else {"rel": 5e-3, "max": 4.4e-2, **differ}
