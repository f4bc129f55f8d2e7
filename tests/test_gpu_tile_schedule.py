"""K and V do not depend on how a launch's tiles are scheduled (units, single tiles, halves and quarters of tiles).

The schedule of the recompute kernel follows the number of 256-row blocks: row counts on either side of its changes
(less than one round of tiles, last rounds of under a quarter, under a half and more, many rounds) are rebuilt from the
store and compared, bit for bit, with the same rows rebuilt in short calls; those are compared with the oracle
elsewhere.
"""
import pytest
import torch

import paper_2603_19664_b200 as kvd
from kvd_synth import GEMMA3_4B_GLOBAL, QWEN3_4B, LayerShape, make_residuals
from gpu_util import dev, open_layer

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [GEMMA3_4B_GLOBAL, QWEN3_4B], ids=lambda s: s.name)
def test_rows_have_the_same_bits_under_every_schedule(shape):
    T, step, kdim = 12000, 2000, shape.n_kv_heads * shape.d_head
    ctx, _ = open_layer(shape, max_tokens=T, with_store=True)
    x = dev(make_residuals(shape, 500, seed=6)).repeat(T // 500, 1)
    ctx.kvd_checkpoint_residual(0, 0, x, torch.arange(T, dtype=torch.int32, device="cuda"), T)
    k, v = (torch.empty((T, kdim), dtype=torch.bfloat16, device="cuda") for _ in range(2))
    for r0 in range(0, T, step):  # 64 tiles, less than one round: whole for the Gemma shape, halves for Qwen's
        ctx.kvd_recompute_kv(0, None, None, step, k[r0:], v[r0:], kdim, seq=0, first_row=r0)
    for n in (1, 257, 1100, 2304, 2305, 2817, 3400, 4737, 5100, 6757, 7168, 8100, 12000):
        kk, vv = (torch.full((n + 1, kdim), 7.0, dtype=torch.bfloat16, device="cuda") for _ in range(2))
        first = T - n if n % 2 else 0
        ctx.kvd_recompute_kv(0, None, None, n, kk, vv, kdim, seq=0, first_row=first)
        assert torch.equal(kk[:n], k[first:first + n]) and torch.equal(vv[:n], v[first:first + n]), n
        assert bool((kk[n] == 7).all()) and bool((vv[n] == 7).all()), n
    assert ctx.kvd_poll_status() == kvd.KVD_OK
    ctx.close()


def test_products_have_the_same_bits_under_every_schedule():
    k = 256
    ctx, _ = open_layer(GEMMA3_4B_GLOBAL, max_tokens=2048)
    g = torch.Generator(device="cuda").manual_seed(3)
    x = torch.randn((1500, k), generator=g, device="cuda").bfloat16()
    for n in (256, 2560, 5120):  # 1 to 120 tiles
        lin = ctx.kvd_scaffold_linear_create((torch.randn((k, n), generator=g, device="cuda") * 0.05).bfloat16(), None, k, n)
        ref = torch.empty((1500, lin.out_cols), dtype=torch.bfloat16, device="cuda")
        for r0 in range(0, 1500, 60):
            ctx.kvd_scaffold_linear(lin, x[r0:], 60, ref[r0:], lin.out_cols)
        for m in (65, 300, 1000, 1500):
            out = torch.empty((m, lin.out_cols), dtype=torch.bfloat16, device="cuda")
            ctx.kvd_scaffold_linear(lin, x, m, out, lin.out_cols)
            assert torch.equal(out, ref[:m]), (n, m)
    assert ctx.kvd_poll_status() == kvd.KVD_OK
    ctx.close()


HEADS64 = LayerShape("h64", 1024, 16, 8, 64, 1e-6, True, 1.0e4)  # four 64-wide heads per 256-column tile


@pytest.mark.parametrize("dtype", [0, 1, 2], ids=["bf16", "f16", "f32"])
@pytest.mark.parametrize("shape", [GEMMA3_4B_GLOBAL, QWEN3_4B, HEADS64], ids=lambda s: s.name)
def test_cut_tiles_have_the_bits_of_whole_ones(shape, dtype):
    """Every element type and head size against calls whose tiles are whole (112 tiles: units of two), from one range and
    from several ranges of two sequences with caller rows beside them."""
    t, kdim = (torch.bfloat16, torch.float16, torch.float32)[dtype], shape.n_kv_heads * shape.d_head
    n_blocks = 2 * kdim // 256
    step = 256 * 112 // n_blocks
    T = 2 * step
    desc = kvd.make_desc(1, shape.d_hidden, shape.n_q_heads, shape.n_kv_heads, shape.d_head, shape.rms_eps, shape.qk_norm,
                         shape.rms_eps, shape.rope_style, 2, T, 1)
    ctx = kvd.Kvd(desc)
    ctx.kvd_set_dtype(dtype)
    g = torch.Generator(device="cuda").manual_seed(8)
    w = (torch.randn((shape.d_hidden, 2 * kdim), generator=g, device="cuda") * 0.02).to(t)
    gammas = [(1 + 0.1 * torch.randn((n,), generator=g, device="cuda")).to(t) for n in (shape.d_hidden, shape.d_head)]
    ctx.kvd_set_layer(0, w, gammas[0], gammas[1] if shape.qk_norm else None, shape.rope_theta)
    arena = torch.empty(kvd.kvd_store_bytes_dtype(desc, 1, dtype), dtype=torch.uint8, device="cuda")
    ctx.kvd_attach_store(arena, 1)
    x = torch.randn((T, shape.d_hidden), generator=g, device="cuda").to(t)
    pos = torch.arange(T, dtype=torch.int32, device="cuda")
    for seq in (0, 1):
        ctx.kvd_checkpoint_residual(seq, 0, x, pos, T)
    k, v = (torch.empty((T, kdim), dtype=t, device="cuda") for _ in range(2))
    for r0 in (0, step):
        ctx.kvd_recompute_kv(0, None, None, step, k[r0:], v[r0:], kdim, seq=0, first_row=r0)
    row_blocks = {8: (1, 3, 7, 9, 10, 12, 14, 19, 20, 28), 4: (1, 5, 9, 18, 19, 23, 28, 37, 38, 56)}[n_blocks]
    for n in [256 * b - 5 for b in row_blocks]:  # rounds of 0 to 3, last rounds of under a quarter, under a half and more
        kk, vv = (torch.full((n + 1, kdim), 7.0, dtype=t, device="cuda") for _ in range(2))
        ctx.kvd_recompute_kv(0, None, None, n, kk, vv, kdim, seq=1, first_row=3)
        assert torch.equal(kk[:n], k[3:n + 3]) and torch.equal(vv[:n], v[3:n + 3]), n
        assert bool((kk[n] == 7).all()) and bool((vv[n] == 7).all()), n
    for scale in (1, 2):  # 11 and 19 (or 20) row blocks over four sources
        ranges = [(0, 5, 1000 * scale), (1, 100, 700 * scale), (0, 2000, 600 * scale)]
        outs = [tuple(torch.full((n, kdim), 7.0, dtype=t, device="cuda") for _ in range(2)) for _, _, n in ranges]
        kk, vv = (torch.full((3, kdim), 7.0, dtype=t, device="cuda") for _ in range(2))
        ctx.kvd_recompute_kv_step(0, [r + o for r, o in zip(ranges, outs)], x[50:], pos[50:], 3, kk, vv, kdim)
        for (_, first, n), (ko, vo) in zip(ranges, outs):
            assert torch.equal(ko, k[first:first + n]) and torch.equal(vo, v[first:first + n]), (first, n)
        assert torch.equal(kk, k[50:53]) and torch.equal(vv, v[50:53])
    assert ctx.kvd_poll_status() == kvd.KVD_OK
    ctx.close()
