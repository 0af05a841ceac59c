"""The decode-attention kernel that takes two units per step, at sizes where the dispatch chooses it (checked): right after a
flush, in fused steps across a flush, and which kernel the other sizes get."""
import pytest
import torch

import gpu_util as U
from paper_2512_19206_b200 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def binding():
    from paper_2512_19206_b200 import build
    build.build()
    from paper_2512_19206_b200 import binding as b
    b.lib()
    return b


def filled(binding, w, **kw):
    cache = U.make_cache(binding, w, extras_budget_bytes=(w.tokens // w.residual_len + 3) * 64 * w.residual_len, **kw)
    for t in range(0, w.tokens, 4096):
        cache.quantize_append(0, *W.tokens(w, 0, t, min(4096, w.tokens - t), device="cuda"))
    return cache


@pytest.mark.parametrize("name,batch,tokens,preset,v_bits", [
    ("qwen7b", 16, 6400, "P24", 2), ("qwen7b", 8, 2560, "P27", 2), ("llama8b", 16, 2560, "P4BASE", 2), ("qwen32b", 16, 2048, "P24", 2),
    ("qwen7b", 16, 6400, "P24", 4), ("qwen7b", 8, 2560, "P27", 4),
])
def test_steps_across_a_flush(binding, name, batch, tokens, preset, v_bits):
    """The window is full: the first step flushes it.  A fused step leaves the state and gives the output of an append and an
    attention call, bit for bit; the attention behind the flush waits before its first read, the others need not."""
    w = W.small(W.CONFIGS[name], n_layers=1, batch=batch, tokens=tokens, **getattr(W, preset))
    a, b = filled(binding, w, v_bits=v_bits), filled(binding, w, v_bits=v_bits)
    for step in range(3):
        k, v, q = [x.contiguous() for x in W.tokens(w, 0, tokens + step, 1, device="cuda")]
        qd = q[:, :, 0].contiguous()
        fused = a.decode_step(0, k, v, q, W.softmax_scale())
        assert a.last_attention() == binding.ATTN_TWO_UNITS | (binding.ATTN_EARLY if step else 0)
        b.quantize_append(0, k, v, q)
        plain = b.decode_attention(0, qd, W.softmax_scale())
        assert b.last_attention() == binding.ATTN_TWO_UNITS | binding.ATTN_EARLY
        assert torch.equal(fused, plain)
        b.written_externally()
        assert torch.equal(b.decode_attention(0, qd, W.softmax_scale()), plain)
        assert b.last_attention() == binding.ATTN_TWO_UNITS
    b.set_attention_kernel(1)
    ref = b.decode_attention(0, qd, W.softmax_scale())
    assert float((plain - ref).abs().max()) <= 4e-3          # both kernels are within 2e-3 of the exact result
    for s in (0, w.batch * w.n_kv_heads - 1):
        assert a.stream_regions(0, s) == b.stream_regions(0, s)
    assert a.status() == b.status() == 0


@pytest.mark.parametrize("name,batch,tokens,R,preset,v_bits,form", [
    ("qwen7b", 8, 390, 128, "P24", 2, 1 + 4), ("qwen7b", 1, 390, 128, "P24", 4, 1), ("qwen7b", 1, 390, 128, "P27", 2, 1),
    ("llama8b", 16, 300, 128, "P27", 4, 1 + 4), ("qwen7b", 1, 450, 128, "P24", 2, 1), ("qwen7b", 8, 8000, 128, "P24", 2, 1),
    ("qwen7b", 8, 16000, 128, "P24", 2, 2), ("qwen7b", 8, 16000, 96, "P24", 2, 1), ("qwen7b", 8, 1000, 128, "P27", 2, 1),
    ("qwen7b", 8, 2000, 128, "P27", 2, 2), ("qwen32b", 32, 1500, 256, "P27", 2, 2 + 4), ("llama8b", 64, 1700, 128, "P4BASE", 4, 1),
    ("llama8b", 64, 1700, 128, "P4BASE", 2, 2),
])
def test_which_kernel(binding, name, batch, tokens, R, preset, v_bits, form):
    w = W.small(W.CONFIGS[name], n_layers=1, batch=batch, tokens=tokens, residual_len=R, group_size=32 if R == 96 else W.CONFIGS[name].group_size,
                **getattr(W, preset))
    cache = filled(binding, w, v_bits=v_bits)
    cache.decode_attention(0, W.decode_query(w, 0, 0, device="cuda"), W.softmax_scale())
    assert cache.last_attention() & 7 == form


@pytest.mark.parametrize("name,batch,tokens,tau16,tau4", [
    ("qwen7b", 16, 6400, 2.5, 1e30), ("qwen32b", 16, 2048, 2.0, 1e30), ("qwen7b", 8, 2560, 2.5, 1.5), ("qwen7b", 8, 2560, 1.0, 0.5),
    ("llama8b", 16, 2560, 0.5, -1.0),
])
def test_more_promoted_channels_than_a_slot_holds(binding, name, batch, tokens, tau16, tau4):
    w = W.small(W.CONFIGS[name], n_layers=1, batch=batch, tokens=tokens, tau_bf16=tau16, tau_u4=tau4)
    cache = U.make_cache(binding, w, extras_budget_bytes=(tokens // 128 + 3) * (128 * 260 + 4096))
    for t in range(0, tokens, 4096):
        cache.quantize_append(0, *W.tokens(w, 0, t, min(4096, tokens - t), device="cuda"))
    n16 = cache.stream_regions(0, 0)["table"][4::8]
    assert max(n16) > 8, n16
    q = W.decode_query(w, 0, 0, device="cuda")
    out = cache.decode_attention(0, q, W.softmax_scale())
    assert cache.last_attention() & 3 == binding.ATTN_TWO_UNITS
    cache.set_attention_kernel(1)
    ref = cache.decode_attention(0, q, W.softmax_scale())
    assert cache.status() == 0
    assert float((out - ref).abs().max()) <= 4e-3          # both kernels are within 2e-3 of the exact result
