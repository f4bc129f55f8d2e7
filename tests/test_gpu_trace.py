"""The trace buffer of kvd_set_trace: a launch that does not fit it records nothing, one that fits stays inside it."""
import pytest
import torch

import paper_2603_19664_b200 as kvd
from kvd_synth import GEMMA3_4B_GLOBAL, QWEN3_4B, make_residuals
from gpu_util import dev, open_layer

pytestmark = pytest.mark.gpu

WORDS = 8 * 16  # int64 slots per CTA


@pytest.mark.parametrize("shape", [QWEN3_4B, GEMMA3_4B_GLOBAL], ids=lambda s: s.name)
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
