"""The trace buffer of kvd_set_trace: a launch that does not fit it records nothing, one that fits stays inside it."""
import dataclasses

import pytest
import torch

import paper_2603_19664_b200 as kvd
from kvd_synth import GEMMA3_4B_GLOBAL, QWEN3_4B, ROPE_HALF, make_residuals
from gpu_util import dev, open_layer
from test_gpu_fused_tail import Step

pytestmark = pytest.mark.gpu

WORDS = 8 * 16  # int64 slots per CTA
GEMMA_HALF = dataclasses.replace(GEMMA3_4B_GLOBAL, name="gemma3-4b-half-split", rope_style=ROPE_HALF)  # (another kernel in short launches)


@pytest.mark.parametrize("shape", [QWEN3_4B, GEMMA3_4B_GLOBAL, GEMMA_HALF], ids=lambda s: s.name)
@pytest.mark.parametrize("n", [65, 200, 256, 300, 2560])
def test_trace_stays_inside_its_buffer(shape, n):
    kdim = shape.n_kv_heads * shape.d_head
    ctx, _ = open_layer(shape, max_tokens=4096)
    desc = kvd.make_desc(1, shape.d_hidden, shape.n_q_heads, shape.n_kv_heads, shape.d_head, shape.rms_eps, shape.qk_norm,
                         shape.rms_eps, shape.rope_style, 1, 4096, 1)
    x = dev(make_residuals(shape, 640, seed=3)).repeat(4, 1)
    pos = torch.arange(2560, dtype=torch.int32, device="cuda")
    k, v, k2, v2 = (torch.empty((n, kdim), dtype=torch.bfloat16, device="cuda") for _ in range(4))
    ctx.kvd_recompute_kv(0, x, pos, n, k, v, kdim)
    words = kvd.kvd_trace_bytes(desc, (n + 255) // 256) // 8
    guard = torch.full((148 * WORDS * 2,), -7, dtype=torch.int64, device="cuda")
    # one CTA's slots short (and half, the size of an uncut launch): nothing is recorded
    for short in (words - WORDS, words // 2):
        ctx.kvd_set_trace(guard[WORDS:WORDS + short])
        ctx.kvd_recompute_kv(0, x, pos, n, k2, v2, kdim)
        assert bool((guard == -7).all()), short
        assert torch.equal(k, k2) and torch.equal(v, v2)
    ctx.kvd_set_trace(guard[WORDS:WORDS + words])
    ctx.kvd_recompute_kv(0, x, pos, n, k2, v2, kdim)
    ctx.kvd_set_trace(None)
    assert torch.equal(k, k2) and torch.equal(v, v2)
    g = guard.cpu().numpy()
    assert (g[:WORDS] == -7).all() and (g[WORDS + words:] == -7).all()
    t = g[WORDS:WORDS + words].reshape(-1, 8, 16)
    assert (t[:, 0, 7] > t[:, 0, 6]).all()  # every CTA recorded its first tile's epilogue
    assert ctx.kvd_poll_status() == kvd.KVD_OK
    ctx.close()


@pytest.mark.parametrize("dtype", [0, 1], ids=["bf16", "f16"])
def test_a_traced_call_of_few_rows(dtype):
    """bf16: a call of at most 64 caller rows takes the kernel that records while a buffer is attached, with the bits of
    the few-row kernel it takes otherwise.  fp16: nothing records, the attached buffer stays untouched."""
    shape = QWEN3_4B
    kdim, t = shape.n_kv_heads * shape.d_head, (torch.bfloat16, torch.float16)[dtype]
    ctx = kvd.Kvd(kvd.make_desc(1, shape.d_hidden, shape.n_q_heads, shape.n_kv_heads, shape.d_head, shape.rms_eps, shape.qk_norm,
                                shape.rms_eps, shape.rope_style, 1, 256, 1))
    ctx.kvd_set_dtype(dtype)
    g = torch.Generator(device="cuda").manual_seed(2)
    w = (torch.randn((shape.d_hidden, 2 * kdim), generator=g, device="cuda") * 0.02).to(t)
    ctx.kvd_set_layer(0, w, torch.ones(shape.d_hidden, device="cuda").to(t), torch.ones(shape.d_head, device="cuda").to(t), shape.rope_theta)
    x, pos = torch.randn((33, shape.d_hidden), generator=g, device="cuda").to(t), torch.arange(33, dtype=torch.int32, device="cuda")
    k, v, k2, v2 = (torch.empty((33, kdim), dtype=t, device="cuda") for _ in range(4))
    ctx.kvd_recompute_kv(0, x, pos, 33, k, v, kdim)
    trace = torch.zeros((148, 8, 16), dtype=torch.int64, device="cuda")
    ctx.kvd_set_trace(trace)
    ctx.kvd_recompute_kv(0, x, pos, 33, k2, v2, kdim)
    ctx.kvd_set_trace(None)
    assert torch.equal(k, k2) and torch.equal(v, v2)
    assert bool((trace[0, 0, 7] > trace[0, 0, 6])) == (dtype == 0) and bool((trace[32:] == 0).all())
    assert ctx.kvd_poll_status() == kvd.KVD_OK
    ctx.close()


@pytest.mark.parametrize("n", [1, 300, 2560, 40000])
def test_a_traced_fused_call_has_the_bits_of_an_untraced_one(n):
    s = Step((4, 2, 256), [n], [[0]], "fp8")
    out = s.run()
    words = kvd.kvd_trace_bytes(s.desc, (n + 255) // 256, 2) // 8
    trace = torch.zeros((words,), dtype=torch.int64, device="cuda")
    s.c.kvd_set_trace(trace)
    traced = s.run()
    s.c.kvd_set_trace(None)
    assert torch.equal(out, traced)
    t = trace.view(-1, 8, 16)
    assert bool((t[:, 0, 7] > t[:, 0, 6]).all())  # every CTA recorded its first tile's epilogue
    s.c.close()
