"""The append path where its shortcuts can go wrong: query magnitudes whose parallel fp64 sum would round (the sum must
then be taken in the defined order), windows of zeros, and the smallest and largest windows and remainders.  Everything
is bit-exact against the oracle."""
import dataclasses

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


def spread(q, kind):
    q = q.float()
    n = q.shape[2]
    if kind == "wide":          # 2^-40 .. 2^40 side by side: the sums need more than 53 bits
        q = q * torch.pow(2.0, 80.0 * ((torch.arange(n) * 7) % 11).float() / 10.0 - 40.0)[None, None, :, None]
    elif kind == "tiny":        # magnitudes below the shortcut's range, subnormals among them
        q = q * 1e-38
    elif kind == "zeros":       # whole channels, whole tokens and whole windows of zeros
        q[..., ::3] = 0.0
        q[:, :, 5::6] = 0.0
        q[:, :, :n // 2] = 0.0
    return q.to(torch.bfloat16)


@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("kind", ["plain", "wide", "tiny", "zeros"])
@pytest.mark.parametrize("R,G,tail", [(32, 32, 1), (128, 64, 128), (256, 128, 200)])
def test_importance_sums(binding, mode, kind, R, G, tail):
    w = W.small(W.CONFIGS["qwen7b"], n_layers=1, batch=1, tokens=3 * R + tail, residual_len=R, group_size=G, **W.P27)
    w = dataclasses.replace(w, tau_bf16=1e-3 if kind == "zeros" else w.tau_bf16)
    k, v, q = W.tokens(w, 0, 0, w.tokens)
    q = spread(q, kind)
    cut = R + 7                 # a bulk part with a tail, then appends that fill the window, flush it and go on in bulk
    cache = U.make_cache(binding, w, importance_mode=mode, extras_budget_bytes=4 * (R * 600 + 512))
    for a, b in ((0, cut), (cut, w.tokens)):
        cache.quantize_append(0, *[x[:, :, a:b].contiguous().cuda() for x in (k, v, q)])
    assert cache.status() == 0
    U.compare_regions(cache, 0, w, U.oracle_streams(w, 0, k, v, q, importance_mode=mode))
