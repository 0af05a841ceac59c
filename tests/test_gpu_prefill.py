"""GPU parity of the prefill call: causal full-precision attention of the prompt against the oracle's plain definition
(within the attention tolerance), and the cache it leaves behind against the oracle's append_many (byte for byte)."""
import numpy as np
import pytest
import torch

import gpu_util as U
from oracle import mixkvq_oracle as O
from paper_2512_19206_b200 import workloads as W

pytestmark = pytest.mark.gpu
ATTN_TOL = 2e-3


@pytest.fixture(scope="module")
def binding():
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2512_19206_b200 import build
    build.build()
    from paper_2512_19206_b200 import binding as b
    b.lib()
    return b


@pytest.mark.parametrize("name,batch,tokens", [("qwen7b", 1, 1), ("qwen7b", 2, 127), ("qwen7b", 1, 128), ("llama8b", 1, 129),
                                               ("qwen7b", 1, 700), ("tiny", 1, 1024)])
def test_prefill_attention_and_cache(binding, name, batch, tokens):
    w = W.small(W.CONFIGS[name], n_layers=1, batch=batch, tokens=tokens, **W.P27)
    k, v, q = W.tokens(w, 0, 0, tokens)
    cache = U.make_cache(binding, w)
    out = cache.prefill(0, k.cuda(), v.cuda(), q.cuda(), W.softmax_scale()).cpu().numpy()
    assert cache.status() == 0
    kf, vf, qf = U.f32(k), U.f32(v), U.f32(q)
    streams = [(0, 0), (batch - 1, w.n_kv_heads - 1)]
    worst = 0.0
    for (b, hk) in set(streams):
        ref = O.causal_attention(qf[b, hk * w.g:(hk + 1) * w.g], kf[b, hk], vf[b, hk], W.softmax_scale())
        worst = max(worst, float(np.abs(out[b, hk * w.g:(hk + 1) * w.g] - ref).max()))
    assert worst <= ATTN_TOL, worst
    assert np.isfinite(out).all()
    U.compare_regions(cache, 0, w, U.oracle_streams(w, 0, k, v, q, streams=list(set(streams))))


@pytest.mark.parametrize("g", [1, 2, 3, 4, 5, 7, 8])
@pytest.mark.parametrize("tokens", [17, 64, 130, 256, 387])
def test_prefill_rows_of_every_group_size(binding, g, tokens):
    """A row tile holds the g heads of neighbouring tokens: groups that end at a key tile's edge or before it, a second group without
    rows, and rows past the prompt, for every g.  Two streams per batch element, so that a row in the wrong place shows."""
    gen = torch.Generator().manual_seed(100 * g + tokens)
    k, v, q = (torch.randn((2, h, tokens, 128), generator=gen).to(torch.bfloat16) for h in (2, 2, 2 * g))
    cache = binding.Cache(binding.make_config(1, 2, 2 * g, 2, tokens, **W.P24))
    out = torch.full((2, 2 * g, tokens, 128), 7.0, device="cuda")
    cache.prefill(0, k.cuda(), v.cuda(), q.cuda(), W.softmax_scale(), out=out)
    assert cache.status() == 0
    qf, kf, vf = (t.double() for t in (q, k.repeat_interleave(g, 1), v.repeat_interleave(g, 1)))
    s = (qf @ kf.transpose(-1, -2)) * W.softmax_scale()
    s.masked_fill_(torch.ones(tokens, tokens).triu(1).bool(), float("-inf"))
    assert float((out.cpu() - torch.softmax(s, -1) @ vf).abs().max()) <= ATTN_TOL


@pytest.mark.parametrize("g,tokens,batch", [(1, 17, 80), (1, 256, 40), (3, 130, 80), (5, 387, 16), (7, 64, 40), (7, 387, 16), (8, 300, 16),
                                            (4, 128, 15), (4, 128, 16), (8, 1, 61), (8, 1, 62)])
def test_prefill_row_tiles_of_256(binding, g, tokens, batch):
    """With more than 123 row tiles (on 148 SMs) a CTA takes 256 rows instead of 128: from 16 sequences of two streams with four tiles on, or from
    62 with one."""
    gen = torch.Generator(device="cuda").manual_seed(100 * g + tokens)
    k, v, q = (torch.randn((batch, h, tokens, 128), generator=gen, device="cuda").to(torch.bfloat16) for h in (2, 2, 2 * g))
    cache = binding.Cache(binding.make_config(1, batch, 2 * g, 2, tokens, **W.P24))
    out = torch.full((batch, 2 * g, tokens, 128), 7.0, device="cuda")
    cache.prefill(0, k, v, q, W.softmax_scale(), out=out)
    assert cache.status() == 0
    qf, kf, vf = (t.double() for t in (q, k.repeat_interleave(g, 1), v.repeat_interleave(g, 1)))
    s = (qf @ kf.transpose(-1, -2)) * W.softmax_scale()
    s.masked_fill_(torch.ones(tokens, tokens, device="cuda").triu(1).bool(), float("-inf"))
    assert float((out - torch.softmax(s, -1) @ vf).abs().max()) <= ATTN_TOL


def test_prefill_large_magnitudes_and_errors(binding):
    w = W.small(W.CONFIGS["qwen7b"], n_layers=1, batch=1, tokens=300)
    k, v, q = W.tokens(w, 0, 0, 300)
    v = (v.float() * 64).to(torch.bfloat16)
    q = (q.float() * 4).to(torch.bfloat16)
    cache = U.make_cache(binding, w)
    out = cache.prefill(0, k.cuda(), v.cuda(), q.cuda(), W.softmax_scale()).cpu().numpy()
    ref = O.causal_attention(U.f32(q)[0, :w.g], U.f32(k)[0, 0], U.f32(v)[0, 0], W.softmax_scale())
    assert float(np.abs(out[0, :w.g] - ref).max()) <= ATTN_TOL * 64
    with pytest.raises(binding.MixKVQError) as e:                      # the layer is no longer empty
        cache.prefill(0, k.cuda(), v.cuda(), q.cuda(), W.softmax_scale())
    assert e.value.code == -2
    cache.reset()
    small = torch.empty(cache.prefill_scratch_bytes(300) - 16, dtype=torch.uint8, device="cuda")
    with pytest.raises(binding.MixKVQError):                           # the scratch buffer is too small
        cache.prefill(0, k.cuda(), v.cuda(), q.cuda(), W.softmax_scale(), scratch=small)
    assert cache.prefill_scratch_bytes(300) == 2 * w.n_kv_heads * 3 * 32768


@pytest.mark.parametrize("sink,mode,v_bits,preset", [(32, 0, 2, "P24"), (0, 1, 2, "P27"), (0, 2, 4, "P24"), (32, 1, 4, "P4BASE")])
def test_prefill_layer_after_layer_with_options(binding, sink, mode, v_bits, preset):
    """Prompts of several layers back to back on one scratch buffer, twice over (the second time on a reset cache): the quantization
    that starts while the attention of its layer still runs leaves the oracle's bytes, with a sink, every importance mode and
    4-bit values, and the outputs repeat themselves."""
    T = 3 * 128 + 45
    w = W.small(W.CONFIGS["qwen7b"], n_layers=3, batch=2, tokens=T, **getattr(W, preset))
    cache = U.make_cache(binding, w, importance_mode=mode, sink_len=sink, v_bits=v_bits, extras_budget_bytes=8 * 64 * 128)
    scratch = torch.empty(cache.prefill_scratch_bytes(T), dtype=torch.uint8, device="cuda")
    data = [W.tokens(w, layer, 0, T) for layer in range(3)]
    cuda = [[x.cuda() for x in d] for d in data]
    outs = []
    for _ in range(2):
        cache.mem.fill_(0xA5)
        cache.reset()
        outs.append([cache.prefill(layer, *cuda[layer], W.softmax_scale(), scratch=scratch) for layer in range(3)])
        assert cache.status() == 0
    for layer in range(3):
        assert torch.equal(outs[0][layer], outs[1][layer])
        streams = [(0, 0), (1, w.n_kv_heads - 1)]
        oracle = U.oracle_streams(w, layer, *data[layer], streams=streams, importance_mode=mode, sink_len=sink, v_bits=v_bits)
        U.compare_regions(cache, layer, w, oracle)
