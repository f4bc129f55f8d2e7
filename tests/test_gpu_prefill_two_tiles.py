"""Long calls of kvd_prefill_attention at d_head 128 take two row tiles per CTA; short ones one.

A token's bits do not depend on the call it is in, so rows of a long call equal the same rows in short calls (which the
other file compares with the oracle): causal and windowed, across a gap between segments, rows past the last key and
before the first one, the last CTA half empty, groups of 1, 2 and 4, bf16 and fp16 (and the same at d_head 64, one tile per CTA).
"""
import numpy as np
import pytest
import torch

import paper_2603_19664_b200 as kvd
from kvd_synth import QWEN3_4B, SMOLLM2_135M, LayerShape, make_layer_weights

pytestmark = pytest.mark.gpu

WINDOW = LayerShape("w128", 128, 16, 16, 128, 1e-6, False, 1.0e4, 300)
PAIRS = LayerShape("g2", 128, 16, 8, 128, 1e-6, False, 1.0e4)


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float16], ids=["bf16", "f16"])
@pytest.mark.parametrize("shape,T,step", [(QWEN3_4B, 1300, 260), (SMOLLM2_135M, 4300, 700), (WINDOW, 2500, 500), (PAIRS, 1500, 300)], ids=lambda v: getattr(v, "name", str(v)))
def test_rows_of_a_long_call_equal_those_of_short_calls(shape, T, step, dtype):
    kdim = shape.n_kv_heads * shape.d_head
    desc = kvd.make_desc(1, shape.d_hidden, shape.n_q_heads, shape.n_kv_heads, shape.d_head, shape.rms_eps, shape.qk_norm,
                         shape.rms_eps, shape.rope_style, 1, T + 64, 1)
    ctx = kvd.Kvd(desc)
    if dtype == torch.float16:
        ctx.kvd_set_dtype(1)
    w = make_layer_weights(shape)

    def dev(bits):  # bf16 bit patterns -> the context's type
        return torch.from_numpy(bits.astype(np.uint32) << np.uint32(16)).view(torch.float32).to(dtype).cuda()

    ctx.kvd_set_layer(0, dev(w.w_kv), dev(w.gamma_in), dev(w.gamma_k) if w.gamma_k is not None else None, shape.rope_theta, shape.sliding_window)
    ws = torch.empty(kvd.kvd_workspace_bytes(desc), dtype=torch.uint8, device="cuda")
    ctx.kvd_attach_workspace(ws)
    g = torch.Generator(device="cuda").manual_seed(17)
    k, v, q = (torch.randn(s, generator=g, device="cuda").to(dtype) for s in ((T, kdim), (T, kdim), (T, shape.n_q_heads, shape.d_head)))
    k *= torch.linspace(0.2, 3.0, T, device="cuda").to(dtype)[:, None]  # growing scores: the reference maximum moves
    cut = T // 2 + 13
    segs = [(k, v, kdim, 3, cut), (k[cut:], v[cut:], kdim, cut + 20, T - cut - 25)]  # positions 3 .. with a gap of 17
    pos = torch.arange(T, dtype=torch.int32, device="cuda")
    out = torch.full_like(q, 9.0)
    ctx.kvd_prefill_attention(0, T, q, pos, segs, 0.0, out)
    part = torch.zeros_like(q[:step])
    for r0 in (0, 1, step + 7, T // 2 - 40, T - step):
        ctx.kvd_prefill_attention(0, step, q[r0:], pos[r0:], segs, 0.0, part)
        assert torch.equal(part, out[r0:r0 + step]), r0
    assert bool((out[:3] == 0).all()) and bool(torch.isfinite(out.float()).all())
    order = torch.randperm(T, generator=g, device="cuda")
    mixed = torch.zeros_like(q)
    ctx.kvd_prefill_attention(0, T, q[order].contiguous(), pos[order].contiguous(), segs, 0.0, mixed)
    assert torch.equal(mixed, out[order])
    assert ctx.kvd_poll_status() == kvd.KVD_OK
    ctx.close()
