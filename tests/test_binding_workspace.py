"""The calls use the tensor that `Cache.workspace` holds when they are made."""
import ctypes as C

import torch

from paper_2512_19206_b200 import binding


class Recorder:
    def __getattr__(self, name):
        return lambda *args: self.calls.append((name, args)) or 0


def test_a_replaced_workspace_is_used(monkeypatch):
    native = Recorder()
    native.calls = []
    monkeypatch.setattr(binding, "_native", native)
    monkeypatch.setattr(binding, "_stream", lambda: 0)
    cache = object.__new__(binding.Cache)
    cache.handle = C.c_void_p(None)
    x = torch.empty(1, 1, 1, 128)
    for n in (64, 4096):
        cache.workspace = torch.empty(n, dtype=torch.uint8)
        cache.decode_attention(0, x, 0.1, out=x)
        cache.decode_step(0, x, x, x, 0.1, out=x)
        cache.rope_decode_step(0, x, x, x, x, x, 3, 0.1, out=x)
        assert [c[0] for c in native.calls] == ["decode_attention", "decode_step", "rope_decode_step"]
        for _, args in native.calls:
            assert args[-3] is cache.workspace and args[-2] == n
        native.calls.clear()


def test_scratch_sizes_beyond_32_bits():
    from paper_2512_19206_b200 import build
    build.build()
    cache = object.__new__(binding.Cache)
    cache.handle = C.c_void_p(None)
    cache.cfg = binding.make_config(1, 16, 32, 8, 131072)
    assert cache.prefill_scratch_bytes(131072) == 2 * 16 * 8 * 1024 * 32768          # 8 GiB
