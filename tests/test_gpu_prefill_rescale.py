"""The prefill attention's lazily raised softmax reference: logits that grow along the prompt (the accumulated output is
rescaled again and again, for some rows of a warp and not for others), shrink, or stay flat, at lengths around the tile edges."""
import math

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


@pytest.mark.parametrize("trend", ["grow", "shrink", "flat"])
@pytest.mark.parametrize("L", [129, 255, 256, 257, 1153])
def test_reference_is_raised(binding, L, trend):
    w = W.small(W.CONFIGS["llama8b"], n_layers=1, batch=1, tokens=L)
    k, v, q = W.tokens(w, 0, 0, L, device="cuda")
    pos = torch.arange(L, device="cuda") / L
    gain = {"grow": 4.0 * pos, "shrink": 4.0 * (1 - pos), "flat": torch.zeros_like(pos)}[trend]
    k = (k.float() * gain[None, None, :, None]).bfloat16()
    cache = U.make_cache(binding, w, extras_budget_bytes=(L // 128 + 2) * 40000)       # many channels are promoted
    out = cache.prefill(0, k, v, q, W.softmax_scale())
    assert cache.status() == 0
    kk, vv = [x.double().repeat_interleave(w.g, 1) for x in (k, v)]
    s = (q.double() @ kk.transpose(2, 3)) * W.softmax_scale()
    s = s.masked_fill(torch.ones(L, L, device="cuda").triu(1).bool(), -math.inf)
    ref = torch.softmax(s, -1) @ vv
    # fp16 probabilities and values: each rounded by at most 2^-11 relative, |v| below 6: 2 * 2^-11 * 6 in the worst case
    assert float((out.double() - ref).abs().max()) <= 6e-3
