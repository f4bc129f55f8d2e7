"""Long calls of kvd_prefill_attention at d_head 128 (more than four 128-row tiles per SM) take two row tiles per CTA,
short ones (at most one per SM) one, those between whichever is estimated to end sooner.

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
@pytest.mark.parametrize("shape,T,step", [(QWEN3_4B, 1300, 260), (SMOLLM2_135M, 4300, 700), (WINDOW, 2500, 500), (PAIRS, 1500, 300), (WINDOW, 5000, 500), (PAIRS, 5000, 300)], ids=lambda v: getattr(v, "name", str(v)))
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


@pytest.mark.parametrize("window", [0, 90])
@pytest.mark.parametrize("group", [1, 2, 3, 4, 8])
def test_a_tile_takes_no_block_that_only_its_neighbour_sees(group, window):
    """A weight of 0 times an infinity in V is a NaN, so an infinity reaches the rows of a 128-row tile through every block
    the tile walks -- and through no other block: as in a call of that tile alone.  A tile without a visible key is zero."""
    n_kv, d_head, first = 8, 128, 5
    shape = LayerShape("inf", 128, group * n_kv, n_kv, d_head, 1e-6, False, 1.0e4, window)
    tok, kdim = 128 // group, n_kv * d_head
    T = tok * (4 * 148 // n_kv + 4) + tok // 2  # more than four tiles per SM: two per CTA; the last one short
    desc = kvd.make_desc(1, shape.d_hidden, shape.n_q_heads, n_kv, d_head, 1e-6, False, 1e-6, shape.rope_style, 1, T + 512, 1)
    ctx = kvd.Kvd(desc)
    w = make_layer_weights(shape)
    bf16 = [torch.from_numpy(b.astype(np.uint32) << np.uint32(16)).view(torch.float32).bfloat16().cuda() for b in (w.w_kv, w.gamma_in)]
    ctx.kvd_set_layer(0, bf16[0], bf16[1], None, shape.rope_theta, window)
    ctx.kvd_attach_workspace(torch.empty(kvd.kvd_workspace_bytes(desc), dtype=torch.uint8, device="cuda"))
    g = torch.Generator(device="cuda").manual_seed(5)
    k, v = (torch.randn((T + 200, kdim), generator=g, device="cuda").bfloat16() for _ in range(2))
    for p in (70, T // 2, T // 2 + 63, T):
        v[p] = float("inf")
    q = torch.randn((T, shape.n_q_heads, d_head), generator=g, device="cuda").bfloat16()
    pos = torch.arange(T, dtype=torch.int32, device="cuda") + 26  # tiles end inside key blocks
    pos[: 2 * tok] = torch.arange(2 * tok, dtype=torch.int32, device="cuda").flip(0) * 2 + first  # two tiles far apart
    pos[4 * tok: 5 * tok] = first - 3  # sees nothing, beside a tile that does
    segs = [(k, v, kdim, first, T + 200)]
    out, alone = torch.full_like(q, 9.0), torch.full_like(q, 9.0)
    ctx.kvd_prefill_attention(0, T, q, pos, segs, 0.0, out)
    for r0 in range(0, T, tok):
        ctx.kvd_prefill_attention(0, min(tok, T - r0), q[r0:], pos[r0:], segs, 0.0, alone[r0:])
    assert ctx.kvd_poll_status() == kvd.KVD_OK
    nan = torch.isnan(alone)
    assert torch.equal(torch.isnan(out), nan) and torch.equal(out[~nan], alone[~nan])
    assert bool(nan.any()) and not bool(nan.all()) and bool((out[4 * tok: 5 * tok] == 0).all())
    ctx.close()
