"""The benchmark's count of split partials against the split itself, CTA by CTA."""
import types

import pytest

import bench
from paper_2512_19206_b200 import workloads as W


@pytest.mark.parametrize("batch,ctas,positions", [(8, 288, 1036), (16, 256, 512), (20, 296, 107), (14, 296, 322), (40, 296, 53), (64, 296, 1000), (1, 56, 29), (18, 144, 40)])
def test_partials_of_a_split(batch, ctas, positions):
    w = W.small(W.CONFIGS["qwen7b" if batch in (8, 1) else "llama8b"], batch=batch)
    streams = w.batch * w.n_kv_heads
    total = positions * streams
    pairs = sum((total * (i + 1) // ctas - 1) // positions - total * i // ctas // positions + 1 for i in range(ctas))
    cache = types.SimpleNamespace(last_attention_ctas=lambda: ctas)
    assert bench.n_split_partials(cache, w, "cpu") == pytest.approx(pairs, rel=0.01)
