"""Precision of the attention outputs beyond what a tolerance on single elements shows: relative error in the 2-norm and bias,
over the lengths where sums are long and where they are split into few parts."""
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


@pytest.mark.parametrize("L", [777, 8192, 32768])
def test_prefill_sum_over_many_tiles(binding, L):
    """Values with a mean, so that a sum that loses something per tile loses it in the same direction every time."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(L)
    k, v, q = [torch.randn((1, 1, L, 128), generator=gen, device="cuda") for _ in range(3)]
    k, v, q = (1.5 * k).bfloat16(), (v.abs() + 0.5).bfloat16(), (1.5 * q).bfloat16()
    w = W.small(W.CONFIGS["tiny"], tokens=L)
    out = U.make_cache(binding, w).prefill(0, k, v, q, W.softmax_scale())
    rows = torch.unique(torch.cat([torch.linspace(0, L - 1, 64).long(), torch.arange(L - 16, L)])).cuda()
    s = (q[:, :, rows].double() @ k.double().transpose(2, 3)) * W.softmax_scale()
    s = s.masked_fill(torch.arange(L, device="cuda") > rows[:, None], -math.inf)
    ref = torch.softmax(s, -1) @ v.double()
    d = out[:, :, rows].double() - ref
    # fp16 probabilities: each rounded to nearest by at most 2^-12 of itself, 2^-12 / sqrt(3) = 1.4e-4 in the root mean square for a
    # row of one dominant token, less where rounding errors average out: 2.8e-5 to 3.9e-5 here.  Rounding to nearest has no
    # bias.  (A tensor-core accumulator that truncates, over the 256 tiles of L = 32768: 1.0e-4 and a bias of -1.4e-4.)
    assert float(d.norm() / ref.norm()) <= 6e-5
    last = slice(-16, None)
    assert abs(float(d[:, :, last].sum() / ref[:, :, last].sum())) <= 4e-5


# Bounds of the relative error in 1e-5, half way between what a reference maximum at the largest probabilities gives (they are
# then exact) and what one anywhere below them by up to a factor of 8 gives (each then rounded by up to 2^-12, and its product
# with the value scale once more).
@pytest.mark.parametrize("name,batch,tokens,preset,v_bits,bound", [
    ("qwen7b", 1, 130, "P27", 2, 9.7),            # 7.2 / 12.2
    ("qwen7b", 8, 390, "P24", 2, 7.9),            # 5.7 / 10.1
    ("qwen7b", 8, 390, "P27", 2, 9.8),            # 6.0 / 13.6
    ("qwen7b", 8, 390, "P24", 4, 8.5),            # 6.2 / 10.7
    ("llama8b", 16, 400, "P4BASE", 2, 8.1),       # 5.6 / 10.6
    ("llama8b", 16, 1200, "P24", 2, 7.7),         # 6.0 / 9.4
    ("qwen7b", 8, 8000, "P24", 2, 4.5),           # 3.8 / 5.3
    ("qwen7b", 8, 8000, "P27", 2, 5.1),           # 4.1 / 6.1
    ("llama8b", 16, 4000, "P4BASE", 2, 10.0),     # 6.9 / 13.0
    ("llama8b", 16, 4000, "P24", 4, 9.5),         # 6.7 / 12.3
    ("qwen32b", 64, 700, "P27", 2, 13.6),         # 10.9 / 16.3
])
def test_decode_probabilities(binding, name, batch, tokens, preset, v_bits, bound):
    """Against the plain-ALU kernel, which is fp32 throughout, on the same cache: one CTA per stream, few and many positions per
    CTA, one and two units per step."""
    w = W.small(W.CONFIGS[name], n_layers=1, batch=batch, tokens=tokens, **getattr(W, preset))
    cache = U.make_cache(binding, w, v_bits=v_bits, extras_budget_bytes=(tokens // 128 + 3) * 64 * 128)
    for t in range(0, tokens, 4096):
        cache.quantize_append(0, *W.tokens(w, 0, t, min(4096, tokens - t), device="cuda"))
    num = den = 0.0
    for step in range(4):
        q = W.decode_query(w, 0, step, device="cuda")
        cache.set_attention_kernel(0)
        out = cache.decode_attention(0, q, W.softmax_scale()).double()
        cache.set_attention_kernel(1)
        ref = cache.decode_attention(0, q, W.softmax_scale()).double()
        num += float((out - ref).square().sum())
        den += float(ref.square().sum())
    assert cache.status() == 0
    assert (num / den) ** 0.5 <= bound * 1e-5
