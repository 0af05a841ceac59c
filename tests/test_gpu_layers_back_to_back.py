"""Decode steps of several layers enqueued back to back, with no other kernel and no wait between them, where the merge of one layer lets
the next layer's split kernel start before its own wait: the same bits as with a synchronization after every call."""
import pytest
import torch

import gpu_util as U
from paper_2512_19206_b200 import workloads as W

pytestmark = pytest.mark.gpu
LAYERS, STEPS = 3, 6


@pytest.fixture(scope="module")
def binding():
    from paper_2512_19206_b200 import build
    build.build()
    from paper_2512_19206_b200 import binding as b
    b.lib()
    return b


@pytest.mark.parametrize("rotate", [False, True])
@pytest.mark.parametrize("preset,lens", [
    ("P24", [23 * 128 + 126] * 16), ("P27", [23 * 128 + 126] * 16), ("P4BASE", [23 * 128 + 125] * 16),
    ("P24", [23 * 128 + 126 - 67 * b for b in range(15)] + [23 * 128 + 124]),      # ragged, windows that fill in different steps
])
def test_steps_of_several_layers(binding, preset, lens, rotate):
    batch, top = len(lens), max(lens)
    w = W.small(W.CONFIGS["llama8b"], n_layers=LAYERS, batch=batch, tokens=top, **getattr(W, preset))
    caches = [U.make_cache(binding, w, extras_budget_bytes=(top // 128 + 4) * 128 * 64) for _ in range(2)]
    for layer in range(LAYERS):
        kvq = W.tokens(w, layer, 0, top, device="cuda")
        for c in caches:
            c.quantize_append_ragged(layer, *kvq, lens)
    ang = torch.arange(top + STEPS + 1, dtype=torch.float64)[:, None] * torch.pow(10000.0, -torch.arange(64, dtype=torch.float64) / 64)
    cos, sin = ang.cos().float().cuda(), ang.sin().float().cuda()
    # the inputs of all calls are there before the first one (a rotating step writes its own)
    inputs = [[[[x.contiguous().clone() for x in W.tokens(w, layer, top + step, 1, device="cuda")] for layer in range(LAYERS)] for step in range(STEPS)]
              for _ in caches]
    outs = [torch.zeros((STEPS, LAYERS, batch, w.n_q_heads, 128), device="cuda") for _ in caches]
    rows = [[list(step.unbind(0)) for step in o.unbind(0)] for o in outs]
    torch.cuda.synchronize()
    for which, cache in enumerate(caches):
        for step in range(STEPS):
            for layer in range(LAYERS):
                k, v, q = inputs[which][step][layer]
                if rotate:
                    cache.rope_decode_step(layer, k, v, q, cos, sin, top + step, W.softmax_scale(), out=rows[which][step][layer])
                else:
                    cache.decode_step(layer, k, v, q, W.softmax_scale(), out=rows[which][step][layer])
                if which == 1:
                    torch.cuda.synchronize()
        torch.cuda.synchronize()
    assert caches[0].last_attention_ctas() > 148 and not caches[0].last_attention() & binding.ATTN_DIRECT      # (a split with a merge that lets go early)
    assert torch.equal(*outs)
    for a, b in zip(*inputs):
        assert all(torch.equal(x, y) for la, lb in zip(a, b) for x, y in zip(la, lb))
    for layer in range(LAYERS):
        for s in (0, 61, batch * w.n_kv_heads - 1):
            assert caches[0].stream_regions(layer, s) == caches[1].stream_regions(layer, s)
    assert caches[0].status() == caches[1].status() == 0
