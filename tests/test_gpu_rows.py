"""The projection of a few rows (at most 64 caller rows, nothing from the store) has the bits of the 256-row tiles.

K and V of n caller rows, and the dense products of at most 64 rows, run on a kernel of their own (narrow tiles over
all SMs).  What they are compared with is the recompute kernel on the same rows inside a larger call, which the other
files compare with the oracle: equality is exact.  Row counts lie around the multiples of 8 and 16 and at the ends of
the range, column counts give narrow, ragged and several tiles per SM.
"""
import numpy as np
import pytest
import torch

import paper_2603_19664_b200 as kvd
from paper_2603_19664_b200.binding import KVD_ERR_POSITION
from kvd_synth import GEMMA3_4B_GLOBAL, QWEN3_4B, SMOLLM2_135M, make_residuals, with_style
from gpu_util import dev, open_layer

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("style", [0, 1])
@pytest.mark.parametrize("shape", [GEMMA3_4B_GLOBAL, QWEN3_4B, SMOLLM2_135M], ids=lambda s: s.name)
def test_few_caller_rows_have_the_bits_of_the_large_call(shape, style):
    shape = with_style(shape, style)
    T, kdim = 200, shape.n_kv_heads * shape.d_head
    ctx, _ = open_layer(shape, max_tokens=1024, max_seqs=2, with_store=True)
    x = dev(make_residuals(shape, T, seed=5))
    pos = (torch.arange(T, dtype=torch.int32, device="cuda") * 5) % 1024
    k, v = (torch.empty((T, kdim), dtype=torch.bfloat16, device="cuda") for _ in range(2))
    ctx.kvd_recompute_kv(0, x, pos, T, k, v, kdim)
    stride = kdim + 8
    for r0, n in ((0, 1), (3, 7), (9, 8), (20, 9), (31, 16), (50, 17), (64, 33), (101, 63), (136, 64)):
        kk, vv = (torch.full((n + 1, stride), 7.0, dtype=torch.bfloat16, device="cuda") for _ in range(2))
        ctx.kvd_recompute_kv(0, x[r0:], pos[r0:], n, kk, vv, stride)
        assert torch.equal(kk[:n, :kdim], k[r0:r0 + n]) and torch.equal(vv[:n, :kdim], v[r0:r0 + n]), (r0, n)
        assert bool((kk[:n, kdim:] == 7).all()) and bool((kk[n] == 7).all()) and bool((vv[n] == 7).all()), (r0, n)
        # the same through the decode step call, which also checkpoints the rows: the store then yields the same K/V
        ctx.kvd_reset_sequence(1)
        ctx.kvd_decode_step_kv(0, [], kdim, x[r0:], pos[r0:], n, [1] * n, kk, vv, stride)
        assert torch.equal(kk[:n, :kdim], k[r0:r0 + n]) and torch.equal(vv[:n, :kdim], v[r0:r0 + n]), (r0, n)
        ks, vs = (torch.empty((n, kdim), dtype=torch.bfloat16, device="cuda") for _ in range(2))
        ctx.kvd_recompute_kv(0, None, None, n, ks, vs, kdim, seq=1, first_row=0)
        assert torch.equal(ks, k[r0:r0 + n]) and torch.equal(vs, v[r0:r0 + n]), (r0, n)
    assert ctx.kvd_poll_status() == kvd.KVD_OK
    bad = torch.full((3,), 4096, dtype=torch.int32, device="cuda")  # past the rotation table: reported and clamped
    ctx.kvd_recompute_kv(0, x, bad, 3, k, v, kdim)
    assert ctx.kvd_poll_status() == KVD_ERR_POSITION
    ctx.close()


@pytest.mark.parametrize("k,n", [(64, 128), (192, 2048), (2560, 2560), (704, 5000), (256, 20480), (320, 40000)])
def test_products_of_few_rows_have_the_bits_of_the_large_call(k, n):
    ctx, _ = open_layer(GEMMA3_4B_GLOBAL, max_tokens=256)
    g = torch.Generator(device="cuda").manual_seed(k + n)
    w = (torch.randn((k, n), generator=g, device="cuda") * 0.05).bfloat16()
    gamma = (1 + 0.1 * torch.randn((k,), generator=g, device="cuda")).bfloat16()
    x = torch.randn((100, k), generator=g, device="cuda").bfloat16()
    for norm in (None, gamma):
        lin = ctx.kvd_scaffold_linear_create(w, norm, k, n, 1e-6)
        big = torch.empty((100, lin.out_cols), dtype=torch.bfloat16, device="cuda")
        ctx.kvd_scaffold_linear(lin, x, 100, big, lin.out_cols)
        for r0, m, pad in ((0, 1, 0), (5, 8, 8), (11, 16, 16), (30, 17, 0), (36, 64, 8)):
            out = torch.full((m + 1, lin.out_cols + pad), 7.0, dtype=torch.bfloat16, device="cuda")
            ctx.kvd_scaffold_linear(lin, x[r0:r0 + m], m, out, lin.out_cols + pad)
            assert torch.equal(out[:m, :lin.out_cols], big[r0:r0 + m]), (r0, m, pad)
            assert bool((out[:m, lin.out_cols:] == 7).all()) and bool((out[m] == 7).all()), (r0, m, pad)
    assert ctx.kvd_poll_status() == kvd.KVD_OK
    ctx.close()


@pytest.mark.parametrize("k,n", [(64, 128), (128, 20480), (256, 20480)])
def test_successive_products_overlap_without_changing_bits(k, n):
    """Launches that follow one another directly, each a dependent of the last, with much tensor memory and little shared
    memory per CTA: every one ends, with the bits of a launch alone."""
    ctx, _ = open_layer(GEMMA3_4B_GLOBAL, max_tokens=256)
    g = torch.Generator(device="cuda").manual_seed(k + n)
    lin = ctx.kvd_scaffold_linear_create((torch.randn((k, n), generator=g, device="cuda") * 0.05).bfloat16(), None, k, n)
    x = torch.randn((8, 5, k), generator=g, device="cuda").bfloat16()
    alone, out = (torch.zeros((8, 5, lin.out_cols), dtype=torch.bfloat16, device="cuda") for _ in range(2))
    for i in range(8):
        ctx.kvd_scaffold_linear(lin, x[i], 5, alone[i], lin.out_cols)
        torch.cuda.synchronize()
    for i in range(8):
        ctx.kvd_scaffold_linear(lin, x[i], 5, out[i], lin.out_cols)
    assert torch.equal(alone, out)
    assert ctx.kvd_poll_status() == kvd.KVD_OK
    ctx.close()


@pytest.mark.parametrize("shape", [GEMMA3_4B_GLOBAL, QWEN3_4B, SMOLLM2_135M], ids=lambda s: s.name)
def test_few_fp16_rows_have_the_bits_of_the_large_call(shape):
    kdim, t = shape.n_kv_heads * shape.d_head, torch.float16
    ctx = kvd.Kvd(kvd.make_desc(1, shape.d_hidden, shape.n_q_heads, shape.n_kv_heads, shape.d_head, shape.rms_eps, shape.qk_norm,
                                shape.rms_eps, shape.rope_style, 1, 1024, 1))
    ctx.kvd_set_dtype(1)
    g = torch.Generator(device="cuda").manual_seed(4)
    w = (torch.randn((shape.d_hidden, 2 * kdim), generator=g, device="cuda") * 0.02).to(t)
    gammas = [(1 + 0.1 * torch.randn((n,), generator=g, device="cuda")).to(t) for n in (shape.d_hidden, shape.d_head)]
    ctx.kvd_set_layer(0, w, gammas[0], gammas[1] if shape.qk_norm else None, shape.rope_theta)
    x = torch.randn((200, shape.d_hidden), generator=g, device="cuda").to(t)
    pos = (torch.arange(200, dtype=torch.int32, device="cuda") * 5) % 1024
    k, v = (torch.empty((200, kdim), dtype=t, device="cuda") for _ in range(2))
    ctx.kvd_recompute_kv(0, x, pos, 200, k, v, kdim)
    for r0, n in ((0, 1), (3, 8), (20, 9), (31, 16), (50, 17), (64, 33), (136, 64)):
        kk, vv = (torch.full((n + 1, kdim + 8), 7.0, dtype=t, device="cuda") for _ in range(2))
        ctx.kvd_recompute_kv(0, x[r0:], pos[r0:], n, kk, vv, kdim + 8)
        assert torch.equal(kk[:n, :kdim], k[r0:r0 + n]) and torch.equal(vv[:n, :kdim], v[r0:r0 + n]), (r0, n)
        assert bool((kk[:n, kdim:] == 7).all()) and bool((kk[n] == 7).all()) and bool((vv[n] == 7).all()), (r0, n)
    assert ctx.kvd_poll_status() == kvd.KVD_OK
    ctx.close()
