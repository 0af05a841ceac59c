"""Timed cases of the MixKVQ cache: what a serving program has it do, through `binding.Cache`.

Every case is one shape of one of these passes:

  decode   one generation step of the whole stack: for every layer `decode_step` (or `rope_decode_step`), the new
           token's append (with the quantizing flush once every R steps) fused with attention over the cache
  attend   `decode_attention` alone, for programs that append and attend in separate calls or replay a graph
  prefill  a new prompt: `reset`, then for every layer `prefill` (causal attention of the prompt, prompt into the cache)
  append   a new prompt whose attention the program does itself: `reset`, then for every layer `quantize_append` of the
           prompt in chunks
  request  a short conversation from start to end: `reset`, `prefill` of the prompt, then decode steps

Shapes are those of `workloads.CONFIGS` and of bench.py, with fewer layers where all of them would only repeat the
same launches.  Inputs follow the recipe of `workloads.py` (N(0,1) in bf16, four outlier key channels per KV head scaled
by 10 to 30, query gains log-uniform in [0.5, 4]), drawn on the GPU from the seed.
"""
from __future__ import annotations

import math

import torch

from paper_2512_19206_b200 import binding, workloads

D = 128
SCALE = workloads.softmax_scale()
FILL_CHUNK = 4096            # tokens per bulk append while a cache is being filled
STEP_INPUTS = 32             # distinct decode-step inputs per layer, used in turn
GROW = 4096                  # decode steps a cache has room for beyond its starting length

# Query and KV heads of the model shapes in workloads.CONFIGS.
SHAPES = {"qwen7b": (28, 4), "llama8b": (32, 8), "qwen32b": (40, 8), "tiny": (1, 1)}
# Threshold presets, and the promoted (BF16) and UINT4 channels per block that they give on this distribution.
PRESETS = {"P24": (workloads.P24, 4, 0), "P27": (workloads.P27, 4, 22), "P4BASE": (workloads.P4BASE, 4, 124)}


def _case(**kw):
    c = dict(kind="decode", model="qwen7b", layers=4, batch=8, tokens=32768, R=128, G=32, preset="P24", v_bits=2,
             sink=0, importance=0, rope=False, steps=0, lens="")
    c.update(kw)
    return c


def listed():
    return [
        # a lone short sequence on the smallest configuration: nothing but latency and launches
        _case(name="attend-tiny", kind="attend", model="tiny", layers=1, batch=1, tokens=1024),
        # one user's chat turn: a short odd prompt, then an answer of a hundred tokens (one flush per layer on the way)
        _case(name="request-chat", kind="request", layers=8, batch=1, tokens=333, steps=100),
        # a small batch at a few thousand tokens with the optional settings: 4-bit values, a sink, cumulative importance
        _case(name="decode-options", model="llama8b", layers=16, batch=4, tokens=6001, G=64, v_bits=4, sink=32,
              importance=1),
        # the benchmark's shape: 7B model, batch 8, 32K tokens, all layers
        _case(name="decode-7b", layers=28),
        # three tiers (the 2.7-bit mix) at an odd length, keys and queries rotated by the call
        _case(name="decode-three-tiers", layers=14, tokens=20011, preset="P27", rope=True),
        # 4-bit base precision on the 8B shape
        _case(name="decode-4bit-base", model="llama8b", layers=8, batch=16, tokens=16384, preset="P4BASE"),
        # a serving batch of unequal lengths
        _case(name="decode-ragged", layers=28, lens="32768,29000,23500,17000,12345,9000,4097,640"),
        # late in a long chain of thought: few sequences, very long
        _case(name="decode-long", layers=8, batch=4, tokens=120000, rope=True),
        # the large model at batch 64: the most cache bytes per launch
        _case(name="decode-32b", model="qwen32b", layers=3, batch=64, G=128),
        # a small batch of short, odd prompts
        _case(name="prefill-short", kind="prefill", model="llama8b", layers=8, batch=4, tokens=777),
        # one long prompt
        _case(name="prefill-long", kind="prefill", layers=1, batch=1, tokens=32768),
        # prompts of a batch, chunk by chunk, quantized only
        _case(name="append-prompts", kind="append", layers=4, batch=8, tokens=8100),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["decode", "decode", "decode", "decode", "ragged", "attend", "prefill", "append", "request"])
    model = rng.choice(["qwen7b", "llama8b", "qwen32b"])
    hkv = SHAPES[model][1]
    preset = rng.choice(["P24", "P24", "P27", "P4BASE"])
    G = rng.choice([32, 32, 32, 64, 128])
    R = rng.choice([128, 128, 128, 32, 64, 256])
    R = max(R, G)
    opts = dict(model=model, preset=preset, G=G, R=R, v_bits=rng.choice([2, 2, 2, 4]), sink=rng.choice([0, 0, 32]),
                importance=rng.choice([0, 0, 0, 1]))
    if kind in ("decode", "ragged"):
        tokens = _log_int(rng, 600, 120000)
        batch = max(1, min(64, int(_log_int(rng, 1, 64) * min(1.0, 500000.0 / (tokens * 64)) + 0.5)))
        # as many layers as make a pass of about the listed ones' bytes, at most a whole small model's
        layers = max(1, min(28, int(5e6 / (batch * hkv * tokens) + 0.5)))
        if kind == "decode":
            return _case(layers=layers, batch=batch, tokens=tokens, rope=rng.random() < 0.5, **opts)
        batch = max(2, batch)
        lens = sorted((_log_int(rng, 500, tokens) for _ in range(batch)), reverse=True)
        return _case(layers=layers, batch=batch, tokens=max(lens), lens=",".join(map(str, lens)), **opts)
    if kind == "attend":
        tokens = _log_int(rng, 200, 60000)
        batch = _log_int(rng, 1, 8)
        return _case(kind="attend", layers=max(1, min(28, int(2e6 / (batch * hkv * tokens)))), batch=batch, tokens=tokens, **opts)
    if kind == "prefill":
        tokens = _log_int(rng, 100, 24000)
        batch = max(1, min(8, 8000 // tokens))
        return _case(kind="prefill", layers=max(1, min(8, 8000 // (tokens * batch))), batch=batch, tokens=tokens, **opts)
    if kind == "append":
        tokens = _log_int(rng, 200, 16000)
        batch = max(1, min(16, 64000 // tokens))
        return _case(kind="append", layers=max(1, min(8, 200000 // (tokens * batch))), batch=batch, tokens=tokens, **opts)
    return _case(kind="request", layers=rng.randint(2, 8), batch=_log_int(rng, 1, 8), tokens=_log_int(rng, 20, 1500),
                 steps=_log_int(rng, 8, 128), **opts)


# ------------------------------------------------------------------------------------------------------- inputs
class _Inputs:
    """Seeded keys, values and queries of a case, on the GPU; the gains belong to (layer, head, channel)."""

    def __init__(self, case, seed):
        self.hq, self.hkv = SHAPES[case["model"]]
        self.gen = torch.Generator(device="cuda")
        self.gen.manual_seed(seed)
        gains = []
        host = torch.Generator()
        host.manual_seed(seed)
        for _ in range(case["layers"]):
            gk = torch.ones(self.hkv, D)
            for h in range(self.hkv):
                chans = torch.randperm(D, generator=host)[:4]
                gk[h, chans] = 10.0 + 20.0 * torch.rand(4, generator=host)
            gq = (0.5 * torch.pow(8.0, torch.rand(self.hkv, D, generator=host))).repeat_interleave(self.hq // self.hkv, 0)
            gq = gq * (0.8 + 0.45 * torch.rand(self.hq, 1, generator=host))
            gains.append((gk[:, None].cuda(), gq[:, None].cuda()))
        self.gains = [(gk.bfloat16(), gq.bfloat16()) for gk, gq in gains]

    def tokens(self, layer, batch, n):
        def normal(heads):
            return torch.empty((batch, heads, n, D), dtype=torch.bfloat16, device="cuda").normal_(generator=self.gen)
        gk, gq = self.gains[layer]
        return normal(self.hkv).mul_(gk), normal(self.hkv), normal(self.hq).mul_(gq)


def _lens(case):
    return [int(x) for x in case["lens"].split(",")] if case["lens"] else [case["tokens"]] * case["batch"]


def _make_cache(case, max_tokens):
    hq, hkv = SHAPES[case["model"]]
    preset = PRESETS[case["preset"]][0]
    budget = 0
    if case["preset"] == "P4BASE":       # a dense high plane per block: the default arena is too small for it
        budget = (max_tokens // case["R"] + 3) * 64 * case["R"]
    cfg = binding.make_config(case["layers"], case["batch"], hq, hkv, max_tokens, residual_len=case["R"],
                              group_size=case["G"], v_bits=case["v_bits"], sink_len=case["sink"],
                              importance_mode=case["importance"], extras_budget_bytes=budget, **preset)
    cache = binding.Cache(cfg)
    cache.mem.zero_()                    # never-written bytes compare equal
    return cache


def _regions(cache):
    """Views of everything the cache stores, over all layers: block tables, packed blocks, promoted channels, residual
    windows, accumulators and sinks."""
    d0 = cache.describe(0)
    layers, streams = cache.cfg.n_layers, d0.n_streams
    layer_stride = cache.describe(1).state_off - d0.state_off if layers > 1 else 0

    def view(off, stride, n):
        return cache.mem.as_strided((layers, streams, n), (layer_stride, stride, 1), off)
    got = [view(d0.state_off, d0.state_stride, 1152), view(d0.table_off, d0.table_stride, 8 * d0.max_blocks),
           view(d0.resk_off, d0.resk_stride, d0.resk_stride), view(d0.resv_off, d0.resv_stride, d0.resv_stride),
           view(d0.base_off, d0.base_stride, d0.base_stride), view(d0.extras_off, d0.extras_stride, d0.extras_stride)]
    if d0.sink_len:
        got.append(view(d0.sink_off, d0.sink_stride, d0.sink_stride))
    return got


def _fill(s):
    """Brings the cache to the case's starting length."""
    case, cache, lens = s["case"], s["cache"], _lens(s["case"])
    inp = _Inputs(case, s["seed"])
    cache.reset()
    for layer in range(case["layers"]):
        for t in range(0, max(lens), FILL_CHUNK):
            n = min(FILL_CHUNK, max(lens) - t)
            k, v, q = inp.tokens(layer, case["batch"], n)
            if case["lens"]:
                cache.quantize_append_ragged(layer, k, v, q, [min(max(x - t, 0), n) for x in lens])
            else:
                cache.quantize_append(layer, k, v, q)
    return inp


def prepare(case, seed):
    L, B, T = case["layers"], case["batch"], case["tokens"]
    hq, hkv = SHAPES[case["model"]]
    kind = case["kind"]
    s = {"case": case, "seed": seed, "kind": kind, "layers": range(L), "at": 0}
    s["out"] = torch.empty((L, B, hq, D), dtype=torch.float32, device="cuda")
    s["out_rows"] = list(s["out"].unbind(0))
    if kind in ("decode", "attend"):
        s["cache"] = _make_cache(case, max(_lens(case)) + GROW)
        inp = _fill(s)
        s["left"] = GROW
    else:
        inp = _Inputs(case, seed)
        s["cache"] = _make_cache(case, T + case["steps"])
    if kind in ("decode", "request"):
        n = STEP_INPUTS if kind == "decode" else case["steps"]
        per_layer = []
        for layer in range(L):
            kvq = [x.permute(2, 0, 1, 3).contiguous().unsqueeze(3).unbind(0) for x in inp.tokens(layer, B, n)]
            per_layer.append(list(zip(*kvq)))
        s["steps"] = list(zip(*per_layer))             # [step][layer] -> k, v [B,Hkv,1,128], q [B,Hq,1,128]
    if kind == "attend":
        s["queries"] = [inp.tokens(layer, B, 1)[2].view(B, hq, D) for layer in range(L)]
    if case["rope"]:
        pos = torch.arange(T + GROW + 1, device="cuda", dtype=torch.float64)
        ang = pos[:, None] * torch.pow(10000.0, -torch.arange(64, device="cuda", dtype=torch.float64) / 64)
        s["cos"], s["sin"] = ang.cos().float(), ang.sin().float()
    if kind in ("prefill", "request"):
        s["prompts"] = [inp.tokens(layer, B, T) for layer in range(L)]
        s["prompt_out"] = [torch.empty((B, hq, T, D), dtype=torch.float32, device="cuda") for _ in range(L)]
        s["scratch"] = torch.empty(s["cache"].prefill_scratch_bytes(T), dtype=torch.uint8, device="cuda")
    if kind == "append":
        s["chunks"] = [[inp.tokens(layer, B, min(FILL_CHUNK, T - t)) for t in range(0, T, FILL_CHUNK)] for layer in range(L)]
    s["regions"] = _regions(s["cache"])
    return s


def _decode(s):
    if s["left"] == 0:                   # the cache is full: the sequences end and new ones take their place
        _fill(s)
        s["left"], s["at"] = GROW, 0
    cache, out, row = s["cache"], s["out_rows"], s["steps"][s["at"] % STEP_INPUTS]
    if s["case"]["rope"]:
        pos, cos, sin = s["case"]["tokens"] + s["at"], s["cos"], s["sin"]
        for layer in s["layers"]:
            k, v, q = row[layer]
            cache.rope_decode_step(layer, k, v, q, cos, sin, pos, SCALE, out=out[layer])
    else:
        for layer in s["layers"]:
            k, v, q = row[layer]
            cache.decode_step(layer, k, v, q, SCALE, out=out[layer])
    s["at"] += 1
    s["left"] -= 1
    return [s["out"]] + s["regions"]


def _attend(s):
    cache, out, queries = s["cache"], s["out_rows"], s["queries"]
    for layer in s["layers"]:
        cache.decode_attention(layer, queries[layer], SCALE, out=out[layer])
    return s["out"]


def _prompt(s):
    cache = s["cache"]
    cache.reset()
    for layer in s["layers"]:
        k, v, q = s["prompts"][layer]
        cache.prefill(layer, k, v, q, SCALE, out=s["prompt_out"][layer], scratch=s["scratch"])


def _prefill(s):
    _prompt(s)
    return s["prompt_out"] + s["regions"]


def _append(s):
    cache = s["cache"]
    cache.reset()
    for layer in s["layers"]:
        for k, v, q in s["chunks"][layer]:
            cache.quantize_append(layer, k, v, q)
    return s["regions"]


def _request(s):
    _prompt(s)
    cache, out = s["cache"], s["out_rows"]
    for row in s["steps"]:
        for layer in s["layers"]:
            k, v, q = row[layer]
            cache.decode_step(layer, k, v, q, SCALE, out=out[layer])
    return s["prompt_out"] + [s["out"]] + s["regions"]


_RUN = {"decode": _decode, "attend": _attend, "prefill": _prefill, "append": _append, "request": _request}


def run(state):
    return _RUN[state["kind"]](state)


# --------------------------------------------------------------------------------------------- work and tolerance
def _packed_token_bytes(case):
    """Bytes of one packed token of one KV head: key codes at their tiers, value codes, scales and zero-points, and the
    token's share of its block's table entry and channel lists."""
    _, n16, n4 = PRESETS[case["preset"]]
    G, R, n2 = case["G"], case["R"], D - n16 - n4
    return (2 * n16 + n4 / 2 + n2 / 4 + 4 * (n4 + n2) / G + 160 / R) + (D * case["v_bits"] / 8 + 4 * D / G)


def _attention_work(case, length, new):
    """(bytes, flops) of decode attention over one sequence of `length` tokens in one layer; `new`: with the step's own
    token stored as well."""
    hq, hkv = SHAPES[case["model"]]
    sink = min(case["sink"], length)
    res = min(length - sink, (length - sink - 1) % case["R"] + 1) if length > sink else 0
    packed = length - sink - res
    per_head = packed * _packed_token_bytes(case) + (sink + res) * 512.0 + (512 * 2 + 2 * 1024 if new else 0)
    return hkv * per_head + hq * D * (2 + 4), 4.0 * D * hq * length


def _append_bytes(case, length):
    """Bytes of putting one sequence's prompt into one layer: keys, values and queries read, the stored form written."""
    hq, hkv = SHAPES[case["model"]]
    sink = min(case["sink"], length)
    res = (length - sink - 1) % case["R"] + 1 if length > sink else 0
    return 256.0 * length * (2 * hkv + hq) + hkv * ((length - sink - res) * _packed_token_bytes(case) + (sink + res) * 512.0)


def work(case):
    L, B, T = case["layers"], case["batch"], case["tokens"]
    hq, _ = SHAPES[case["model"]]
    nbytes = flops = 0.0
    if case["kind"] in ("decode", "attend"):
        for x in _lens(case):
            b, f = _attention_work(case, x + (1 if case["kind"] == "decode" else 0), case["kind"] == "decode")
            nbytes += L * b
            flops += L * f
    if case["kind"] in ("append", "prefill", "request"):
        nbytes += L * B * _append_bytes(case, T)
    if case["kind"] in ("prefill", "request"):
        nbytes += L * B * hq * T * D * 4.0
        flops += L * B * hq * 4.0 * D * T * (T + 1) / 2
    if case["kind"] == "request":
        for i in range(case["steps"]):
            b, f = _attention_work(case, T + i + 1, True)
            nbytes += L * B * b
            flops += L * B * f
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    if case["kind"] == "append":
        return "exact"                   # codes, scales, channel lists, windows, sums of magnitudes: defined bit for bit
    # Attention outputs: probabilities (and in decode their products with the value scales) are fp16, everything else is
    # exact or fp32.  Against the library's fp32 plain-ALU kernel (decode) and fp64 attention (prefill) the listed cases
    # show rel 0.5e-4 to 1.8e-4 and max 0.1e-3 to 1.8e-3: four times that.  The stored bytes that come back beside the
    # outputs are whole numbers and have to be the same.
    return {"rel": 7e-4, "max": 8e-3}
