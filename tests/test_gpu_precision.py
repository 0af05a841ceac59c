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
