"""The native form of the per-token calls: argument checks on CPU, the same results as the library's own entry on the GPU."""
import ctypes as C

import pytest
import torch

from paper_2512_19206_b200 import binding, workloads as W


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2512_19206_b200 import build
    build.build()


def test_the_module_is_built_for_this_interpreter():
    import sysconfig

    from paper_2512_19206_b200 import build
    assert build.CALLS.endswith(sysconfig.get_config_var("EXT_SUFFIX")) and binding._calls().__file__ == build.CALLS


def test_arguments_are_checked():
    n = binding._calls()
    assert n.decode_step(None, 0, None, None, None, None, 0.1, None, 0, None) == -1
    assert n.decode_attention(None, 0, None, None, 1, None, 0, 0) == -1
    assert n.rope_decode_step(None, 0, None, None, None, None, None, 3, None, 0.1, None, 0, 0) == -1
    assert n.quantize_append(None, 0, None, None, None, 1, 0) == -1
    with pytest.raises(TypeError):
        n.decode_attention(None, 0)
    with pytest.raises(TypeError):
        n.quantize_append(None, "0", None, None, None, 1, 0)
    with pytest.raises(AssertionError):                     # a CPU tensor
        n.quantize_append(None, 0, torch.empty(2), None, None, 1, 0)
    with pytest.raises(AttributeError):                     # an address is not a tensor
        n.quantize_append(None, 0, 256, None, None, 1, 0)


@pytest.mark.gpu
def test_native_calls_pass_every_argument_on():
    w = W.small(W.CONFIGS["qwen7b"], n_layers=2, batch=2, tokens=200, **W.P27)
    cfg = binding.make_config(w.n_layers, w.batch, w.n_q_heads, w.n_kv_heads, 1024, tau_bf16=w.tau_bf16, tau_u4=w.tau_u4)
    k, v, q = (t.cuda() for t in W.tokens(w, 1, 0, w.tokens + 1))
    cos, sin = torch.rand(256, 64, device="cuda"), torch.rand(256, 64, device="cuda")
    scale, L, p = W.softmax_scale(), binding.lib(), binding._ptr
    outs, regions = [], []
    for native in (True, False):
        cache = binding.Cache(cfg)
        prompt = [t[:, :, :-1].contiguous() for t in (k, v, q)]
        kn, vn, qn = (t[:, :, -1:].clone().contiguous() for t in (k, v, q))
        qd = qn[:, :, 0].contiguous()
        out = [torch.empty(qd.shape, dtype=torch.float32, device="cuda") for _ in range(3)]
        st, s = binding._stream(), C.c_float(scale)
        if native:
            cache.quantize_append(1, *prompt)
            cache.decode_attention(1, qd, scale, out[0])
            cache.decode_step(1, kn, vn, qn, scale, out[1])
            cache.rope_decode_step(1, kn, vn, qn, cos, sin, 17, scale, out[2])
        else:
            h, ws = cache.handle, cache._ws
            assert L.mixkvq_quantize_append(h, 1, *map(p, prompt), w.tokens, st) == 0
            assert L.mixkvq_decode_attention(h, 1, p(qd), p(out[0]), s, *ws, st) == 0
            assert L.mixkvq_decode_step(h, 1, p(kn), p(vn), p(qn), p(out[1]), s, *ws, st) == 0
            assert L.mixkvq_rope_decode_step(h, 1, p(kn), p(vn), p(qn), p(cos), p(sin), 17, p(out[2]), s, *ws, st) == 0
        assert cache.status() == 0
        outs.append(out + [kn, qn])
        regions.append([cache.stream_regions(1, i) for i in range(w.batch * w.n_kv_heads)])
    assert all(torch.equal(a, b) for a, b in zip(*outs))    # the same launches on the same bytes
    assert regions[0] == regions[1]
