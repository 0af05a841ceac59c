"""The decode-attention kernel that takes two units per step (chosen for larger caches) against the library's plain-ALU fp32
kernel on the same cache: group sizes, block sizes, tier mixes (promoted and UINT4 channels beyond what a step's staging
holds among them), 4-bit values, sequences that end anywhere, and a ragged batch."""
import pytest
import torch

import gpu_util as U
from paper_2512_19206_b200 import workloads as W

pytestmark = pytest.mark.gpu
# both kernels are within 2e-3 of the exact result (tests/test_gpu_parity.py), so they are within 4e-3 of each other
TOL = 4e-3


@pytest.fixture(scope="module")
def binding():
    from paper_2512_19206_b200 import build
    build.build()
    from paper_2512_19206_b200 import binding as b
    b.lib()
    return b


@pytest.mark.parametrize("tokens,R,G,preset,v_bits,budget", [
    (6400, 128, 32, "P24", 2, (0, 0)), (6400 + 33, 64, 64, "P24", 2, (0, 0)), (6400 + 127, 256, 128, "P24", 2, (0, 0)),
    (6400 + 1, 128, 128, "P24", 2, (0, 0)), (6400 + 77, 128, 32, "P27", 2, (0, 0)), (6400, 128, 32, "P4BASE", 2, (0, 0)),
    (6400 + 64, 128, 64, "P24", 4, (0, 0)), (6400, 128, 32, "P27", 4, (0, 0)), (6400, 64, 32, "P4BASE", 4, (0, 0)),
    (6400, 128, 32, "P24", 2, (8, 0)), (6400, 128, 32, "P24", 2, (21, 0)), (6400, 128, 32, "P24", 2, (3, 45)),
    (6400, 64, 32, "P24", 2, (13, 32)),
])
def test_two_units_per_step(binding, tokens, R, G, preset, v_bits, budget):
    w = W.small(W.CONFIGS["qwen7b"], n_layers=1, batch=16, tokens=tokens, residual_len=R, group_size=G, **getattr(W, preset))
    cache = U.make_cache(binding, w, v_bits=v_bits, budget_bf16=budget[0], budget_u4=budget[1],
                         extras_budget_bytes=(tokens // R + 4) * R * 128)
    for t in range(0, tokens, 3200):
        cache.quantize_append(0, *W.tokens(w, 0, t, min(3200, tokens - t), device="cuda"))
    q = W.decode_query(w, 0, 0, device="cuda")
    out = cache.decode_attention(0, q, W.softmax_scale())
    cache.set_attention_kernel(1)
    ref = cache.decode_attention(0, q, W.softmax_scale())
    assert cache.status() == 0
    assert float((out - ref).abs().max()) <= TOL


def test_two_units_per_step_ragged(binding):
    # every sequence of the batch alone in a cache of its own gives the same result
    lens = [12000, 64, 9001, 0, 128, 16123, 8000, 7777, 129, 16000, 9000, 14000, 1, 15999, 12345, 13000]
    w = W.small(W.CONFIGS["qwen7b"], n_layers=1, batch=16, tokens=max(lens))
    k, v, q = W.tokens(w, 0, 0, max(lens), device="cuda")
    cache = U.make_cache(binding, w)
    cache.quantize_append_ragged(0, k, v, q, lens)
    qd = W.decode_query(w, 0, 0, device="cuda")
    out = cache.decode_attention(0, qd, W.softmax_scale())
    one = W.small(w, batch=1)
    for b, n in enumerate(lens):
        if n == 0:
            assert float(out[b].abs().max()) == 0.0
            continue
        c = U.make_cache(binding, one)
        c.quantize_append(0, *[x[b:b + 1, :, :n].contiguous() for x in (k, v, q)])
        c.set_attention_kernel(1)
        ref = c.decode_attention(0, qd[b:b + 1].contiguous(), W.softmax_scale())
        assert float((out[b] - ref[0]).abs().max()) <= TOL, b
    assert cache.status() == 0
