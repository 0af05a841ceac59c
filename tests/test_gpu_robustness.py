"""GPU tests of the decode-attention kernel's behaviour off the happy path: a bounded wait that runs out, and the early
request of packed blocks ahead of the stream-order wait."""
import pytest
import torch

import gpu_util as U
from paper_2512_19206_b200 import workloads as W

pytestmark = pytest.mark.gpu
ATTN_TOL = 2e-3


@pytest.fixture(scope="module")
def binding():
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2512_19206_b200 import build
    build.build()
    from paper_2512_19206_b200 import binding as b
    b.lib()
    return b


def _filled(binding, tokens=5 * 128 + 40, **kw):
    w = W.small(W.CONFIGS["qwen7b"], n_layers=1, batch=2, tokens=tokens, **W.P27)
    k, v, q = W.tokens(w, 0, 0, tokens)
    cache = U.make_cache(binding, w, **kw)
    cache.quantize_append(0, k.cuda(), v.cuda(), q.cuda())
    return w, cache, (k, v, q)


def test_a_wait_that_runs_out_returns_with_the_status_bit(binding):
    """The barrier of every pair's first staged copy is armed for 16 bytes more than the copy delivers (the test hook
    of the C ABI), so no wait on it can succeed: every wait gives up after 64 polls, the call returns, the status word
    says so and the output is zero.  After a reset the same cache works again."""
    w, cache, (k, v, q) = _filled(binding)
    qd = W.decode_query(w, 0, 0).cuda()
    want = cache.decode_attention(0, qd, W.softmax_scale())
    assert cache.status() == 0
    cache.test_arm_copy_timeout(16, 64)
    got = cache.decode_attention(0, qd, W.softmax_scale())
    torch.cuda.synchronize()                                   # the call came back
    assert cache.status() & binding.DEV_COPY_TIMEOUT
    assert torch.isfinite(got).all()
    # the packed units gave nothing; what is left is the residual window alone, or zero for a stream whose pairs all gave up
    assert float((got - want).abs().max()) > ATTN_TOL
    cache.test_arm_copy_timeout(0, 0)
    cache.reset()
    assert cache.status() == 0
    cache.quantize_append(0, k.cuda(), v.cuda(), q.cuda())
    again = cache.decode_attention(0, qd, W.softmax_scale())
    assert cache.status() == 0
    assert torch.equal(again, want)


def test_a_prefill_wait_that_runs_out_returns_with_the_status_bit(binding):
    """The same for the prefill attention: the barrier of every CTA's first key tile never completes, every role of the
    CTA gives up after 64 polls, the call returns with the status bit and writes no output; after a reset the call works."""
    w = W.small(W.CONFIGS["qwen7b"], n_layers=1, batch=1, tokens=600, **W.P24)
    k, v, q = [t.cuda() for t in W.tokens(w, 0, 0, 600)]
    cache = U.make_cache(binding, w)
    want = cache.prefill(0, k, v, q, W.softmax_scale())
    assert cache.status() == 0
    cache.reset()
    cache.test_arm_copy_timeout(16, 64)
    out = torch.full_like(want, 7.0)
    cache.prefill(0, k, v, q, W.softmax_scale(), out=out)
    torch.cuda.synchronize()                                   # the call came back
    assert cache.status() & binding.DEV_COPY_TIMEOUT
    assert bool((out == 7.0).all())                            # no row was written
    cache.test_arm_copy_timeout(0, 0)
    cache.reset()
    assert cache.status() == 0
    again = cache.prefill(0, k, v, q, W.softmax_scale())
    assert cache.status() == 0
    assert torch.equal(again, want)


def test_attention_right_after_a_flush_and_after_an_external_write(binding):
    """Packed blocks are requested ahead of the stream-order wait except right after a flush of the same layer (or
    when the caller says it wrote cache memory itself); the results do not depend on which path was taken."""
    w, cache, (k, v, q) = _filled(binding, tokens=6 * 128)          # the window is full: the next append flushes
    k1, v1, q1 = W.tokens(w, 0, w.tokens, 1)
    qd = W.decode_query(w, 0, 1).cuda()
    cache.quantize_append(0, k1.cuda(), v1.cuda(), q1.cuda())       # flush + append enqueued directly before the attention
    first = cache.decode_attention(0, qd, W.softmax_scale())        # waits before its first read
    second = cache.decode_attention(0, qd, W.softmax_scale())       # requests its first blocks early
    cache.written_externally()
    third = cache.decode_attention(0, qd, W.softmax_scale())        # waits again
    assert torch.equal(first, second) and torch.equal(first, third)
    kk = torch.cat([k, k1], 2); vv = torch.cat([v, v1], 2); qq = torch.cat([q, q1], 2)
    oracle = U.oracle_streams(w, 0, kk, vv, qq, **{})
    ref = U.oracle_attention(w, oracle, qd.cpu())
    assert U.max_abs_err(w, first, ref) <= ATTN_TOL
    assert cache.status() == 0


@pytest.mark.parametrize("name,batch,tokens,preset,v_bits", [
    ("qwen7b", 16, 6400, "P24", 2),          # two units per step, a logits warp per team
    ("qwen7b", 16, 6400, "P27", 2),          # two logits warps per team
    ("qwen7b", 8, 8000, "P24", 2),           # one unit per step
    ("qwen32b", 64, 700, "P24", 4),          # one unit per step, several streams per CTA
])
def test_a_wait_that_runs_out_with_more_steps_than_stages(binding, name, batch, tokens, preset, v_bits):
    """As above where every team has more units than its ring has stages: after the give-up no stage is refilled, so that every
    copy under way is awaited before the ring is reused; the call returns, and after a reset the cache works again."""
    w = W.small(W.CONFIGS[name], n_layers=1, batch=batch, tokens=tokens, **getattr(W, preset))
    cache = U.make_cache(binding, w, v_bits=v_bits)
    qd = W.decode_query(w, 0, 0, device="cuda")

    def fill():
        for t in range(0, tokens, 4096):
            cache.quantize_append(0, *W.tokens(w, 0, t, min(4096, tokens - t), device="cuda"))
    fill()
    want = cache.decode_attention(0, qd, W.softmax_scale())
    assert cache.status() == 0
    cache.test_arm_copy_timeout(16, 64)
    got = cache.decode_attention(0, qd, W.softmax_scale())
    torch.cuda.synchronize()
    assert cache.status() & binding.DEV_COPY_TIMEOUT
    assert torch.isfinite(got).all()
    cache.test_arm_copy_timeout(0, 0)
    cache.reset()
    fill()
    again = cache.decode_attention(0, qd, W.softmax_scale())
    assert cache.status() == 0
    assert torch.equal(again, want)


def test_a_prefill_wait_for_the_last_values_that_runs_out(binding):
    """A CTA's last value tile never arrives where its number is odd or it is the prompt's last: tiles 1, 3 and 4 of the five.  A row tile
    holds the heads of neighbouring tokens, whose last key tile is the one that they lie in: the rows of the tokens in those tiles need
    the missing product and are left unwritten, all others are right."""
    w = W.small(W.CONFIGS["qwen7b"], n_layers=1, batch=1, tokens=600, **W.P24)
    k, v, q = [t.cuda() for t in W.tokens(w, 0, 0, 600)]
    cache = U.make_cache(binding, w)
    want = cache.prefill(0, k, v, q, W.softmax_scale())
    cache.reset()
    cache.test_arm_value_copy_timeout(16, 2000)
    out = torch.full_like(want, 7.0)
    cache.prefill(0, k, v, q, W.softmax_scale(), out=out)
    torch.cuda.synchronize()
    assert cache.status() & binding.DEV_COPY_TIMEOUT
    for a, b, whole in ((0, 128, True), (128, 256, False), (256, 384, True), (384, 512, False), (512, 600, False)):
        assert torch.equal(out[:, :, a:b], want[:, :, a:b] if whole else torch.full_like(want[:, :, a:b], 7.0)), (a, b)
    cache.test_arm_value_copy_timeout(0, 0)
    cache.reset()
    assert torch.equal(cache.prefill(0, k, v, q, W.softmax_scale()), want)
    assert cache.status() == 0


def test_no_early_request_when_the_last_call_went_to_another_stream(binding):
    """A flush of layer 0 on one stream, a call for layer 1 on another, attention over layer 0 on the first: the flush may still be
    the last thing on that stream, so the attention waits before its first read.  On one stream throughout it need not."""
    w = W.small(W.CONFIGS["qwen7b"], n_layers=2, batch=2, tokens=6 * 128, **W.P24)
    qd = W.decode_query(w, 0, 0, device="cuda")
    outs = []
    for streams in ((0, 0), (0, 1)):
        cache = U.make_cache(binding, w)
        data = [[t.cuda() for t in W.tokens(w, layer, 0, w.tokens + 1)] for layer in (0, 1)]
        for layer in (0, 1):
            cache.quantize_append(layer, *[x[:, :, :-1].contiguous() for x in data[layer]])
        one = [[x[:, :, -1:].contiguous() for x in data[layer]] for layer in (0, 1)]
        torch.cuda.synchronize()
        s = [torch.cuda.Stream(), torch.cuda.Stream()]
        with torch.cuda.stream(s[streams[0]]):
            cache.quantize_append(0, *one[0])                  # the window is full: flushed
        with torch.cuda.stream(s[streams[1]]):
            cache.quantize_append(1, *one[1])
        with torch.cuda.stream(s[streams[0]]):
            outs.append(cache.decode_attention(0, qd, W.softmax_scale()))
        assert bool(cache.last_attention() & binding.ATTN_EARLY) == (streams[0] == streams[1])
        torch.cuda.synchronize()
        assert cache.status() == 0
    assert torch.equal(*outs)
