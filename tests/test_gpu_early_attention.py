"""Attention over a cache, straight behind the projection of the new tokens: its kernels are started before that projection
has ended, and the next step's projection before that attention has, whatever their grids.  Steps made one right after the
other, with nothing between them, give the results of the same steps with the GPU waited for after every call."""
import pytest
import torch

import paper_2603_19664_b200 as kvd
from kvd_synth import GEMMA3_4B_GLOBAL, QWEN3_4B, SMOLLM2_135M, make_layer_weights
from gpu_util import dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [GEMMA3_4B_GLOBAL, QWEN3_4B, SMOLLM2_135M], ids=lambda s: s.name)
@pytest.mark.parametrize("batch,ctx", [(1, 70), (1, 9000), (9, 900), (16, 900), (17, 900), (64, 300)])  # one wave of CTAs to several
def test_attention_sees_the_new_tokens_of_its_own_step(shape, batch, ctx):
    kdim = shape.n_kv_heads * shape.d_head
    w = make_layer_weights(shape)
    desc = kvd.make_desc(1, shape.d_hidden, shape.n_q_heads, shape.n_kv_heads, shape.d_head, shape.rms_eps, shape.qk_norm, shape.rms_eps,
                         shape.rope_style, 1, ctx + 64, batch)
    c = kvd.Kvd(desc)
    c.kvd_set_layer(0, dev(w.w_kv), dev(w.gamma_in), dev(w.gamma_k) if w.gamma_k is not None else None, shape.rope_theta, shape.sliding_window)
    c.kvd_attach_workspace(torch.empty(kvd.kvd_workspace_bytes(desc), dtype=torch.uint8, device="cuda"))
    g = torch.Generator(device="cuda").manual_seed(4)
    k, v = (torch.randn((batch, ctx + 1, kdim), generator=g, device="cuda").bfloat16() for _ in range(2))
    q = torch.randn((batch, shape.n_q_heads, shape.d_head), generator=g, device="cuda").bfloat16()
    xs = (3.0 * torch.randn((12, batch, shape.d_hidden), generator=g, device="cuda")).bfloat16()
    pos = torch.full((batch,), ctx, dtype=torch.int32, device="cuda")
    segs = [[(k[b], v[b], kdim, 0, ctx + 1)] for b in range(batch)]

    def steps(after_each_call):
        """Every step overwrites the new tokens' keys and values, which the step before it reads."""
        outs = [torch.zeros_like(q) for _ in xs]
        k[:, ctx], v[:, ctx] = 0, 0
        torch.cuda.synchronize()
        for x, out in zip(xs, outs):
            c.kvd_decode_step_kv(0, [], kdim, x, pos, batch, None, k[:, ctx], v[:, ctx], (ctx + 1) * kdim)
            after_each_call()
            c.kvd_decode_attention(0, batch, q, [ctx] * batch, segs, 0.0, out)
            after_each_call()
        torch.cuda.synchronize()
        return outs

    chained = steps(lambda: None)
    alone = steps(torch.cuda.synchronize)
    for i, (a, b) in enumerate(zip(chained, alone)):
        assert torch.equal(a, b), i
    assert len({bytes(t.view(torch.uint8).cpu().numpy().tobytes()) for t in alone}) == len(alone)  # (the steps differ)
    assert c.kvd_poll_status() == kvd.KVD_OK
    c.close()
