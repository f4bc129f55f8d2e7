"""Attention at the end of the int range: keys up to the last position a segment may hold (2^31 - 2) and queries at 2^31 - 1
give the bits of the same call moved to small positions by whole blocks; a query at 2^31 - 1 sees every key anywhere."""
import pytest
import torch

import paper_2603_19664_b200 as kvd

pytestmark = pytest.mark.gpu

LAST = 2**31 - 1


@pytest.mark.parametrize("window", [0, 200])
@pytest.mark.parametrize("n_q,n_kv,d_head,rows", [(8, 4, 256, 50), (8, 4, 256, 1300), (32, 8, 128, 30), (32, 8, 128, 700), (32, 8, 128, 3000), (9, 3, 64, 400)])
def test_the_last_positions(n_q, n_kv, d_head, rows, window):
    kdim, T = n_kv * d_head, 64 * 10 - 1
    c = kvd.Kvd(kvd.make_desc(1, 256, n_q, n_kv, d_head, 1e-6, False, 1e-6, 0, 1, 1024, 1))
    g = torch.Generator(device="cuda").manual_seed(rows + window)
    c.kvd_set_layer(0, (torch.randn((256, 2 * kdim), generator=g, device="cuda") * 0.02).bfloat16(), torch.ones(256, device="cuda").bfloat16(), None, 1e4, window)
    c.kvd_attach_workspace(torch.empty(kvd.kvd_workspace_bytes(kvd.make_desc(1, 256, n_q, n_kv, d_head, 1e-6, False, 1e-6, 0, 1, 1024, 1)), dtype=torch.uint8, device="cuda"))
    k, v = (torch.randn((T, kdim), generator=g, device="cuda").bfloat16() for _ in range(2))
    q = torch.randn((rows, n_q, d_head), generator=g, device="cuda").bfloat16()
    pos = torch.randint(0, T + 1, (rows,), generator=g, device="cuda")
    pos[:3] = torch.tensor([T, T - 1, 0])
    outs = []
    for first in (640, LAST - T):  # both multiples of 64
        out = torch.full_like(q, 9.0)
        segs = [(k, v, kdim, first, 300), (k[310:], v[310:], kdim, first + 310, T - 310)]
        c.kvd_prefill_attention(0, rows, q, (pos + first).to(torch.int32), segs, 0.0, out)
        outs.append(out)
    assert torch.equal(outs[0], outs[1]) and bool(torch.isfinite(outs[1].float()).all())
    if window == 0:
        everything, ref = torch.zeros_like(q), torch.zeros_like(q)
        segs = [(k, v, kdim, 3, T)]
        c.kvd_prefill_attention(0, rows, q, torch.full((rows,), T + 2, dtype=torch.int32, device="cuda"), segs, 0.0, ref)
        c.kvd_prefill_attention(0, rows, q, torch.full((rows,), LAST, dtype=torch.int32, device="cuda"), segs, 0.0, everything)
        assert torch.equal(everything, ref)
    one, last = torch.zeros_like(q[:1]), torch.zeros_like(q[:1])
    c.kvd_decode_attention(0, 1, q, [1 << 20], [[(k, v, kdim, (1 << 20) - T, T)]], 0.0, one)
    c.kvd_decode_attention(0, 1, q, [LAST], [[(k, v, kdim, LAST - T, T)]], 0.0, last)
    assert (one.float() - last.float()).norm() <= 1e-2 * one.float().norm()  # (chunks need not start alike)
    assert c.kvd_poll_status() == kvd.KVD_OK
    c.close()
