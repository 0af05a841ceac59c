"""Tokens with NaNs and infinities: the append paths agree with one another and with the definition (the oracle's serial sums)."""
import numpy as np
import pytest
import torch

import gpu_util as U
from oracle import mixkvq_oracle as O
from paper_2512_19206_b200 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def binding():
    from paper_2512_19206_b200 import build
    build.build()
    from paper_2512_19206_b200 import binding as b
    b.lib()
    return b


def queries(q, kind):
    q = q.clone()
    if kind == "nan token":              # nothing else in the append of that token
        q[:, :, 40] = float("nan")
    elif kind == "nan window":           # a window of nothing else
        q[:, :, 32:64] = float("nan")
    elif kind == "nan among zeros":
        q[:, :, :64] = 0.0
        q[:, :, 40, 17] = float("nan")
    elif kind == "infinity":
        q[:, :, 40, ::5] = float("-inf")
    return q


def same(got, want):
    """State of one stream: magnitude sums with NaNs where the oracle has them (their payload is not defined), then the counters."""
    a, b = np.frombuffer(got[:1024], np.float64), np.frombuffer(want[:1024], np.float64)
    return np.array_equal(a, b, equal_nan=True) and got[1024:] == want[1024:]


@pytest.mark.parametrize("path", ["bulk", "single", "step"])
@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("kind", ["nan token", "nan window", "nan among zeros", "infinity"])
def test_query_magnitudes(binding, kind, mode, path):
    T = 2 * 32 + 9
    w = W.small(W.CONFIGS["qwen7b"], n_layers=1, batch=1, tokens=T, residual_len=32, **W.P4BASE)
    k, v, q = W.tokens(w, 0, 0, T)
    q = queries(q, kind)
    cache = U.make_cache(binding, w, importance_mode=mode, extras_budget_bytes=8 * 64 * 128)
    cache.mem.fill_(0xA5)                # whatever is not written shows
    cache.reset()
    cuda = [x.cuda() for x in (k, v, q)]
    if path == "bulk":
        cache.quantize_append(0, *cuda)
    for t in range(T if path != "bulk" else 0):
        x = [y[:, :, t:t + 1].contiguous() for y in cuda]
        if path == "single":
            cache.quantize_append(0, *x)
        else:
            cache.decode_step(0, *x, W.softmax_scale())
    for (b, hk), st in U.oracle_streams(w, 0, k, v, q, importance_mode=mode).items():
        got, want = cache.stream_regions(0, b * w.n_kv_heads + hk), O.pack_stream(st)
        assert same(got["state"], want["state"]), (hk, "state")
        for key in ("table", "base", "extras", "resK", "resV"):
            assert got[key] == want[key], (hk, key)


@pytest.mark.parametrize("tokens", [3 * 128 + 1, 128 * 128])        # one unit per step, two units per step
def test_blocks_without_a_high_plane(binding, tokens):
    """4-bit base with an arena that is too small: the blocks that did not fit have no high plane, and the attention takes
    their codes as the plain-ALU kernel does (the low two bits) without reading behind the arena."""
    w = W.small(W.CONFIGS["qwen7b"], n_layers=1, batch=4, tokens=tokens, **W.P4BASE)
    cache = U.make_cache(binding, w, extras_budget_bytes=2 * 4 * 2048)
    cache.mem.fill_(0xA5)
    cache.reset()
    for t in range(0, tokens, 4096):
        cache.quantize_append(0, *W.tokens(w, 0, t, min(4096, tokens - t), device="cuda"))
    assert cache.status() == binding.DEV_EXTRAS_FULL
    q = W.decode_query(w, 0, 0, device="cuda")
    out = cache.decode_attention(0, q, W.softmax_scale())
    cache.set_attention_kernel(1)
    ref = cache.decode_attention(0, q, W.softmax_scale())
    assert float((out - ref).abs().max()) <= 4e-3          # both kernels are within 2e-3 of the exact result


def elements(x, kind, seed):
    g = torch.Generator().manual_seed(seed)
    x = x.float()
    if kind == "subnormal":              # ranges from 0 to a few units of 2^-133, the last bit of a bf16 subnormal
        scale = torch.pow(2.0, torch.randint(-133, -124, (*x.shape[:2], 1, x.shape[3]), generator=g).float())
        x = torch.randint(0, 24, x.shape, generator=g).float() * scale
    elif kind == "huge":                 # ranges that overflow fp32 among them
        x = x * 2.0 ** 125.5
    else:
        value = {"nan": float("nan"), "inf": float("inf"), "-inf": float("-inf")}[kind]
        x = torch.where(torch.rand(x.shape, generator=g) < 0.002, torch.tensor(value), x)
    return x.to(torch.bfloat16)


def quantize_past_nans(x, bits):
    """The oracle's quantizer with extrema that pass over NaNs and code 0 for what has no quotient, as the header's contract for
    finite values extends to them in the kernels."""
    x = np.asarray(x, np.float32)
    levels = np.float32((1 << bits) - 1)
    with np.errstate(all="ignore"):
        z, mx = np.fmin.reduce(x, axis=-1), np.fmax.reduce(x, axis=-1)
        s = O.bf16_round_up(((mx - z).astype(np.float32) / levels).astype(np.float32))
        y = np.rint(((x - z[..., None]).astype(np.float32) / s[..., None]).astype(np.float32))
    return np.where(np.isnan(y) | (s == 0)[..., None], 0, np.clip(y, 0, float(levels))).astype(np.uint8), s, z


@pytest.mark.parametrize("layout", [0, 1])
@pytest.mark.parametrize("preset,v_bits", [("P24", 2), ("P4BASE", 4)])
@pytest.mark.parametrize("kind", ["subnormal", "huge", "nan", "inf", "-inf"])
def test_codes(binding, monkeypatch, kind, preset, v_bits, layout):
    if layout == 1 and v_bits == 4:
        pytest.skip("the tile layout holds 2-bit values only")
    w = W.small(W.CONFIGS["qwen7b"], n_layers=1, batch=1, tokens=3 * 128 + 5, **{**getattr(W, preset), "tau_bf16": 1e39})
    if preset == "P24":
        w = W.small(w, tau_u4=1e39)
    k, v, q = W.tokens(w, 0, 0, w.tokens)
    k, v = elements(k, kind, 1), elements(v, kind, 2)
    monkeypatch.setattr(O, "quantize_groups", quantize_past_nans)
    monkeypatch.setattr(O, "salience", lambda acc, cnt, kw, bits: (np.ones(128), np.ones(128), np.ones(128)))     # (one tier: 1e39 is infinite in fp32)
    caches = [U.make_cache(binding, w, v_bits=v_bits, layout=layout, extras_budget_bytes=4 * 64 * 128) for _ in range(2)]
    caches[0].quantize_append(0, k.cuda(), v.cuda(), q.cuda())
    for a in range(0, w.tokens, 100):                      # windows that are flushed from the residual store
        caches[1].quantize_append(0, *[x[:, :, a:a + 100].contiguous().cuda() for x in (k, v, q)])
    for cache in caches:
        assert cache.status() == 0
        for (b, hk), st in U.oracle_streams(w, 0, k, v, q, v_bits=v_bits).items():
            got, want = cache.stream_regions(0, hk), O.pack_stream(st, layout=layout)
            for key in ("table", "base", "extras"):
                assert got[key] == want[key], (hk, key)
