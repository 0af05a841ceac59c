"""The decode-attention kernel that writes its output itself (one CTA per stream: small caches, and batches whose streams fill
the GPU) and the split grids on either side of that choice, against the library's plain-ALU fp32 kernel; the partial form
gives the same rows and the log-denominator of the merged call."""
import pytest
import torch

import gpu_util as U
from paper_2512_19206_b200 import workloads as W

pytestmark = pytest.mark.gpu
TOL = 4e-3          # both kernels are within 2e-3 of the exact result (tests/test_gpu_parity.py)


@pytest.fixture(scope="module")
def binding():
    from paper_2512_19206_b200 import build
    build.build()
    from paper_2512_19206_b200 import binding as b
    b.lib()
    return b


@pytest.mark.parametrize("name,batch,tokens,R,preset", [
    ("qwen7b", 1, 1, 128, "P24"), ("qwen7b", 1, 128, 128, "P24"), ("qwen7b", 2, 640, 128, "P24"), ("qwen7b", 2, 900, 128, "P24"),
    ("qwen7b", 2, 300, 128, "P27"), ("qwen7b", 2, 500, 128, "P27"), ("llama8b", 3, 97, 32, "P24"), ("llama8b", 2, 401, 128, "P4BASE"),
    ("qwen32b", 32, 777, 128, "P24"), ("qwen32b", 32, 1500, 256, "P27"), ("qwen32b", 37, 600, 128, "P24"),
])
def test_direct_output(binding, name, batch, tokens, R, preset):
    w = W.small(W.CONFIGS[name], n_layers=1, batch=batch, tokens=tokens, residual_len=R, group_size=32 if R == 32 else W.CONFIGS[name].group_size,
                **getattr(W, preset))
    cache = U.make_cache(binding, w, extras_budget_bytes=(tokens // R + 3) * R * 128)
    cache.quantize_append(0, *W.tokens(w, 0, 0, tokens, device="cuda"))
    q = W.decode_query(w, 0, 0, device="cuda")
    out = cache.decode_attention(0, q, W.softmax_scale())
    part, lse = cache.decode_attention_partial(0, q, W.softmax_scale())
    assert torch.equal(out, part) and bool(torch.isfinite(lse).all())
    merged = binding.merge_partials(torch.stack([part, part]), torch.stack([lse, lse]))      # twice the same set: the same rows
    assert float((merged - out).abs().max()) <= 1e-6 * float(out.abs().max())
    cache.set_attention_kernel(1)
    ref = cache.decode_attention(0, q, W.softmax_scale())
    assert cache.status() == 0
    assert float((out - ref).abs().max()) <= TOL


@pytest.mark.parametrize("name,batch,tokens,preset,v_bits,form", [
    ("qwen7b", 1, 200, "P27", 4, 1 + 4 + 32), ("llama8b", 1, 450, "P24", 2, 1 + 4 + 32), ("llama8b", 1, 560, "P24", 2, 1), ("qwen7b", 16, 511, "P4BASE", 2, 1 + 4 + 32),
    ("qwen7b", 16, 1152, "P27", 2, 2), ("llama8b", 16, 1000, "P24", 4, 1 + 4 + 32), ("llama8b", 18, 200, "P24", 2, 1 + 4), ("llama8b", 19, 700, "P27", 2, 2 + 4),
    ("llama8b", 18, 249, "P24", 2, 1 + 4), ("llama8b", 16, 249, "P27", 2, 1 + 4 + 32), ("qwen7b", 1, 383, "P24", 2, 1 + 4 + 32), ("llama8b", 16, 639, "P4BASE", 4, 1 + 4 + 32),
    ("qwen7b", 8, 249, "P24", 4, 1 + 4 + 32),
])
def test_eight_pairs_per_stream(binding, name, batch, tokens, preset, v_bits, form):
    """One CTA of eight warp pairs per stream while every stream has an SM to itself, on both sides of where that ends (148 SMs: 18
    sequences of the 8b shape) and of the positions up to which it is chosen: more units than pairs, fewer, pairs without a unit; a fused
    step across a flush leaves the same bytes as append and attention."""
    w = W.small(W.CONFIGS[name], n_layers=1, batch=batch, tokens=tokens, **getattr(W, preset))
    caches = [U.make_cache(binding, w, v_bits=v_bits, sink_len=32 if batch == 18 else 0, extras_budget_bytes=(tokens // 128 + 4) * 128 * 128) for _ in range(2)]
    for c in caches:
        c.quantize_append(0, *W.tokens(w, 0, 0, tokens, device="cuda"))
    k, v, q = [x.contiguous() for x in W.tokens(w, 0, tokens, 1, device="cuda")]
    out = caches[0].decode_step(0, k, v, q, W.softmax_scale())
    assert caches[0].last_attention() & ~binding.ATTN_EARLY == form
    caches[1].quantize_append(0, k, v, q)
    plain, lse = caches[1].decode_attention_partial(0, q[:, :, 0].contiguous(), W.softmax_scale())
    assert torch.equal(out, plain) and bool(torch.isfinite(lse).all())
    for s in (0, batch * w.n_kv_heads - 1):
        assert caches[0].stream_regions(0, s) == caches[1].stream_regions(0, s)
    caches[1].set_attention_kernel(1)
    ref = caches[1].decode_attention(0, q[:, :, 0].contiguous(), W.softmax_scale())
    assert caches[0].status() == caches[1].status() == 0
    assert float((out - ref).abs().max()) <= TOL


@pytest.mark.parametrize("name,batch,tokens,preset,v_bits,straddles", [
    ("llama8b", 9, 3000, "P24", 2, False), ("llama8b", 12, 4000, "P27", 2, False), ("llama8b", 16, 2000, "P4BASE", 2, False), ("llama8b", 18, 2000, "P24", 2, False),
    ("llama8b", 20, 3000, "P24", 2, True), ("llama8b", 14, 10000, "P24", 2, True), ("llama8b", 14, 6000, "P24", 4, True), ("qwen7b", 19, 12000, "P27", 2, True),
    ("llama8b", 16, 10000, "P4BASE", 2, True),
])
def test_split_that_straddles_streams(binding, name, batch, tokens, preset, v_bits, straddles):
    """Stream counts that leave many CTA slots idle at a whole number of CTAs per stream: all slots are used and CTAs straddle streams where
    the streams are long enough for it; shorter ones keep a whole number."""
    w = W.small(W.CONFIGS[name], n_layers=1, batch=batch, tokens=tokens, **getattr(W, preset))
    cache = U.make_cache(binding, w, v_bits=v_bits, extras_budget_bytes=(tokens // 128 + 3) * 128 * 64)
    for t in range(0, tokens, 4096):
        cache.quantize_append(0, *W.tokens(w, 0, t, min(4096, tokens - t), device="cuda"))
    q = W.decode_query(w, 0, 0, device="cuda")
    out = cache.decode_attention(0, q, W.softmax_scale())
    assert (cache.last_attention_ctas() % (batch * w.n_kv_heads) != 0) == straddles
    cache.set_attention_kernel(1)
    ref = cache.decode_attention(0, q, W.softmax_scale())
    assert cache.status() == 0
    assert float((out - ref).abs().max()) <= TOL
