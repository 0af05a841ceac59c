"""GPU parity of the rotating append (Appendix D: scores and keys are taken after the rotary embedding): the cache
after mixkvq_rope_append / mixkvq_rope_decode_step equals, byte for byte, the oracle's cache after rotating with the
oracle's rope and appending; the rotated tensors left in place equal the oracle's rotation bit for bit."""
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


def tables(n_pos, base=10000.0):
    inv = base ** (-np.arange(64, dtype=np.float64) / 64)
    ang = np.arange(n_pos, dtype=np.float64)[:, None] * inv[None]
    return np.cos(ang).astype(np.float32), np.sin(ang).astype(np.float32)


def rotate_with_the_oracle(k, v, q, cos, sin, pos0):
    n = k.shape[2]
    kr = O.rope(U.f32(k), cos[pos0:pos0 + n], sin[pos0:pos0 + n])
    qr = O.rope(U.f32(q), cos[pos0:pos0 + n], sin[pos0:pos0 + n])
    return torch.from_numpy(kr).to(torch.bfloat16), v, torch.from_numpy(qr).to(torch.bfloat16)


@pytest.mark.parametrize("layout", [0, 1])
def test_bulk_then_decode_steps_with_rotation(binding, layout):
    w = W.small(W.CONFIGS["qwen7b"], n_layers=1, batch=2, tokens=3 * 128 + 57, **W.P27)
    n_dec = 140                                    # crosses a flush
    cos, sin = tables(w.tokens + n_dec + 8)
    cosd, sind = torch.from_numpy(cos).cuda(), torch.from_numpy(sin).cuda()
    k, v, q = W.tokens(w, 0, 0, w.tokens + n_dec)
    cache = U.make_cache(binding, w, max_tokens=w.tokens + n_dec + 256, layout=layout)
    # bulk append with rotation: the tensors come back rotated
    kd, vd, qd = k[:, :, :w.tokens].contiguous().cuda(), v[:, :, :w.tokens].contiguous().cuda(), q[:, :, :w.tokens].contiguous().cuda()
    cache.rope_append(0, kd, vd, qd, cosd, sind, 0)
    kr, vr, qr = rotate_with_the_oracle(k[:, :, :w.tokens], v[:, :, :w.tokens], q[:, :, :w.tokens], cos, sin, 0)
    assert torch.equal(kd.cpu(), kr) and torch.equal(qd.cpu(), qr)
    ks, vs, qs = [kr], [vr], [qr]
    scale = W.softmax_scale()
    out = None
    for i in range(n_dec):
        t = w.tokens + i
        k1, v1, q1 = k[:, :, t:t + 1].contiguous().cuda(), v[:, :, t:t + 1].contiguous().cuda(), q[:, :, t:t + 1].contiguous().cuda()
        if i % 2 == 0:
            out = cache.rope_decode_step(0, k1, v1, q1, cosd, sind, t, scale)
        else:                                      # the two-call form
            cache.rope_append(0, k1, v1, q1, cosd, sind, t)
            out = cache.decode_attention(0, q1.view(w.batch, w.n_q_heads, 128), scale)
        a, b, c = rotate_with_the_oracle(k[:, :, t:t + 1], v[:, :, t:t + 1], q[:, :, t:t + 1], cos, sin, t)
        assert torch.equal(q1.cpu(), c) and torch.equal(k1.cpu(), a)
        ks.append(a); vs.append(b); qs.append(c)
    kk, vv, qq = torch.cat(ks, 2), torch.cat(vs, 2), torch.cat(qs, 2)
    oracle = U.oracle_streams(w, 0, kk, vv, qq)
    U.compare_regions(cache, 0, w, oracle)
    ref = U.oracle_attention(w, oracle, qq[:, :, -1])
    assert U.max_abs_err(w, out, ref) <= ATTN_TOL
    assert cache.status() == 0


@pytest.mark.parametrize("name,batch,tokens,preset,lens,sink", [
    ("qwen7b", 1, 20, "P24", None, 0),                  # the split kernel writes the output itself, four pairs
    ("llama8b", 20, 300, "P24", None, 0),               # the same with more streams than SMs
    ("qwen32b", 32, 1500, "P27", None, 0),              # the same, two units per step
    ("qwen7b", 1, 1000, "P27", None, 0),                # merge: a CTA per head
    ("qwen7b", 8, 6000, "P4BASE", None, 0),             # the same, two logits warps
    ("llama8b", 16, 1700, "P24", None, 0),              # merge: a CTA per stream
    ("qwen7b", 3, 700, "P24", [700, 128, 5], 0),        # ragged, one window full
    ("qwen7b", 1, 40, "P24", None, 64),                 # room in the sink: append and attention by themselves
])
def test_step_that_rotates_equals_rotation_append_and_attention(binding, name, batch, tokens, preset, lens, sink):
    w = W.small(W.CONFIGS[name], n_layers=1, batch=batch, tokens=tokens, group_size=32, **getattr(W, preset))
    cos, sin = [torch.from_numpy(x).cuda() for x in tables(tokens + 8)]
    caches = [U.make_cache(binding, w, sink_len=sink, extras_budget_bytes=(tokens // 128 + 4) * 128 * 128) for _ in range(2)]
    kvq = W.tokens(w, 0, 0, tokens, device="cuda")
    for c in caches:
        c.quantize_append_ragged(0, *kvq, lens or [tokens] * batch)
    for step in range(2):
        a, b = [[x.contiguous().clone() for x in W.tokens(w, 0, tokens + step, 1, device="cuda")] for _ in range(2)]
        out = caches[0].rope_decode_step(0, *a, cos, sin, tokens + step, W.softmax_scale())
        caches[1].rope_append(0, *b, cos, sin, tokens + step)
        assert torch.equal(out, caches[1].decode_attention(0, b[2].view(batch, w.n_q_heads, 128), W.softmax_scale()))
        assert all(torch.equal(x, y) for x, y in zip(a, b))
    for s in (0, batch * w.n_kv_heads - 1):
        assert caches[0].stream_regions(0, s) == caches[1].stream_regions(0, s)
    assert caches[0].status() == caches[1].status() == 0


@pytest.mark.parametrize("name,batch,tokens,preset,R,G,v_bits,sink,form,straddles", [
    ("qwen7b", 1, 300, "P24", 128, 32, 2, 0, 1 + 4 + 32, False),       # eight pairs of warps
    ("qwen7b", 16, 511, "P4BASE", 128, 64, 4, 0, 1 + 4 + 32, False),
    ("qwen7b", 8, 300, "P27", 128, 128, 2, 32, 1 + 4 + 32, False),
    ("llama8b", 3, 1000, "P27", 32, 32, 4, 0, 1, False),               # one unit per step, blocks of one unit
    ("qwen7b", 2, 700, "P24", 128, 32, 2, 64, 1, False),               # a filled sink
    ("qwen7b", 4, 1000, "P4BASE", 128, 128, 2, 0, 1, False),
    ("llama8b", 20, 3000, "P24", 128, 32, 2, 0, 2, True),              # CTAs that straddle two streams
    ("llama8b", 14, 6000, "P24", 128, 64, 4, 0, 2, True),
    ("llama8b", 40, 700, "P27", 128, 32, 2, 0, 2, True),               # CTAs with several streams
    ("llama8b", 40, 700, "P24", 64, 32, 4, 0, 1, True),
    ("qwen7b", 8, 6000, "P27", 128, 128, 4, 0, 2, False),              # two units per step
    ("qwen32b", 32, 1500, "P4BASE", 256, 128, 2, 32, 2 + 4, False),    # the same, output written by the split kernel
])
def test_step_that_rotates_in_every_form_of_the_split_kernel(binding, name, batch, tokens, preset, R, G, v_bits, sink, form, straddles):
    """Bit for bit the rotation, the append and the attention as calls of their own; a second step rotates again from the caller's rows."""
    w = W.small(W.CONFIGS[name], n_layers=1, batch=batch, tokens=tokens, residual_len=R, group_size=G, **getattr(W, preset))
    cos, sin = [torch.from_numpy(x).cuda() for x in tables(tokens + 8)]
    caches = [U.make_cache(binding, w, sink_len=sink, v_bits=v_bits, extras_budget_bytes=(tokens // R + 4) * R * 128) for _ in range(2)]
    for t in range(0, tokens, 2048):
        kvq = W.tokens(w, 0, t, min(2048, tokens - t), device="cuda")
        for c in caches:
            c.quantize_append(0, *kvq)
    for step in range(2):
        a, b = [[x.contiguous().clone() for x in W.tokens(w, 0, tokens + step, 1, device="cuda")] for _ in range(2)]
        out = caches[0].rope_decode_step(0, *a, cos, sin, tokens + step, W.softmax_scale())
        assert caches[0].last_attention() & ~binding.ATTN_EARLY == form
        assert (caches[0].last_attention_ctas() % (batch * w.n_kv_heads) != 0) == straddles
        caches[1].rope_append(0, *b, cos, sin, tokens + step)
        assert torch.equal(out, caches[1].decode_attention(0, b[2].view(batch, w.n_q_heads, 128), W.softmax_scale()))
        assert all(torch.equal(x, y) for x, y in zip(a, b))
    for s in (0, batch * w.n_kv_heads // 2, batch * w.n_kv_heads - 1):
        assert caches[0].stream_regions(0, s) == caches[1].stream_regions(0, s)
    assert caches[0].status() == caches[1].status() == 0


def test_rotation_errors(binding):
    w = W.small(W.CONFIGS["qwen7b"], n_layers=1, batch=1, tokens=40)
    cos, sin = tables(64)
    cosd, sind = torch.from_numpy(cos).cuda(), torch.from_numpy(sin).cuda()
    k, v, q = W.tokens(w, 0, 0, 40)
    cache = U.make_cache(binding, w, max_tokens=32)
    kd, qd = k.cuda(), q.cuda()
    with pytest.raises(binding.MixKVQError) as e:
        cache.rope_append(0, kd, v.cuda(), qd, cosd, sind, 0)         # more tokens than the cache holds
    assert e.value.code == -5
    assert torch.equal(kd.cpu(), k) and torch.equal(qd.cpu(), q)        # nothing was rotated
    lib = binding.lib()
    assert lib.mixkvq_rope_append(None, 0, None, None, None, None, None, 0, 1, None) == -1
