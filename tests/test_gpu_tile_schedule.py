"""K and V do not depend on how a launch's tiles are scheduled (units, single tiles, halves and quarters of tiles).

The schedule of the recompute kernel follows the number of 256-row blocks: row counts on either side of its changes
(less than one round of tiles, last rounds of under a quarter, under a half and more, many rounds) are rebuilt from the
store and compared, bit for bit, with the same rows rebuilt in short calls; those are compared with the oracle
elsewhere.
"""
import pytest
import torch

import paper_2603_19664_b200 as kvd
from kvd_synth import GEMMA3_4B_GLOBAL, QWEN3_4B, make_residuals
from gpu_util import dev, open_layer

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [GEMMA3_4B_GLOBAL, QWEN3_4B], ids=lambda s: s.name)
def test_rows_have_the_same_bits_under_every_schedule(shape):
    T, step, kdim = 12000, 2000, shape.n_kv_heads * shape.d_head
    ctx, _ = open_layer(shape, max_tokens=T, with_store=True)
    x = dev(make_residuals(shape, 500, seed=6)).repeat(T // 500, 1)
    ctx.kvd_checkpoint_residual(0, 0, x, torch.arange(T, dtype=torch.int32, device="cuda"), T)
    k, v = (torch.empty((T, kdim), dtype=torch.bfloat16, device="cuda") for _ in range(2))
    for r0 in range(0, T, step):  # 64 tiles: one per cluster
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
