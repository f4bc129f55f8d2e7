"""Attention over a cache, straight behind the projection of the new tokens: its kernels are started before that projection
has ended, whatever their grid.  The result is that of the same call made after the GPU was waited for, step after step."""
import pytest
import torch

import paper_2603_19664_b200 as kvd
from kvd_synth import GEMMA3_4B_GLOBAL, QWEN3_4B, make_layer_weights
from gpu_util import dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [GEMMA3_4B_GLOBAL, QWEN3_4B], ids=lambda s: s.name)
@pytest.mark.parametrize("batch,ctx", [(1, 70), (1, 9000), (16, 900), (17, 900), (64, 300)])  # one wave of CTAs to several
def test_attention_sees_the_new_tokens_of_its_own_step(shape, batch, ctx):
    kdim = shape.n_kv_heads * shape.d_head
    w = make_layer_weights(shape)
    desc = kvd.make_desc(1, shape.d_hidden, shape.n_q_heads, shape.n_kv_heads, shape.d_head, shape.rms_eps, shape.qk_norm, shape.rms_eps,
                         shape.rope_style, 1, ctx + 64, batch)
    c = kvd.Kvd(desc)
    c.kvd_set_layer(0, dev(w.w_kv), dev(w.gamma_in), dev(w.gamma_k), shape.rope_theta, shape.sliding_window)
    c.kvd_attach_workspace(torch.empty(kvd.kvd_workspace_bytes(desc), dtype=torch.uint8, device="cuda"))
    g = torch.Generator(device="cuda").manual_seed(4)
    k, v = (torch.randn((batch, ctx + 1, kdim), generator=g, device="cuda").bfloat16() for _ in range(2))
    q = torch.randn((batch, shape.n_q_heads, shape.d_head), generator=g, device="cuda").bfloat16()
    xs = (3.0 * torch.randn((12, batch, shape.d_hidden), generator=g, device="cuda")).bfloat16()
    pos = torch.full((batch,), ctx, dtype=torch.int32, device="cuda")
    segs = [[(k[b], v[b], kdim, 0, ctx + 1)] for b in range(batch)]
    outs = [torch.zeros_like(q) for _ in xs]
    news = []
    for x, out in zip(xs, outs):
        c.kvd_decode_step_kv(0, [], kdim, x, pos, batch, None, k[:, ctx], v[:, ctx], (ctx + 1) * kdim)
        c.kvd_decode_attention(0, batch, q, [ctx] * batch, segs, 0.0, out)
        news.append((k[:, ctx].clone(), v[:, ctx].clone()))
    again = torch.zeros_like(q)
    for (kn, vn), out in zip(news, outs):
        k[:, ctx], v[:, ctx] = kn, vn
        torch.cuda.synchronize()
        c.kvd_decode_attention(0, batch, q, [ctx] * batch, segs, 0.0, again)
        assert torch.equal(again, out)
    assert c.kvd_poll_status() == kvd.KVD_OK
    c.close()
