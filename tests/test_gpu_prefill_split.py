"""Calls of kvd_prefill_attention whose tiles leave half of the SMs idle (d_head 128 and 256, six key blocks or more): a tile
is shared by two CTAs.  A row's bits do not depend on that: they equal those of the same rows inside a call of more tiles
than that, which takes whole tiles, and (in the other file) follow the oracle.

Walks of 0 to 13 blocks and of 79 (every remainder of the four blocks the CTAs take turns by, and many rounds of every
ring), growing scores (the reference maximum moves, the accumulated output is rescaled), blocks across a gap between
segments, windows, every group size, one tile to 74, tiles with empty rows, rows without a key, rows past the call, fp16.
"""
import pytest
import torch

import paper_2603_19664_b200 as kvd

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", [0, 1], ids=["bf16", "f16"])
@pytest.mark.parametrize("window", [0, 450])
@pytest.mark.parametrize("n_q,n_kv,d_head", [(8, 4, 256), (4, 4, 256), (6, 2, 256), (16, 2, 256), (32, 8, 128), (4, 4, 128), (6, 2, 128), (8, 1, 128)])
def test_a_shared_tile_has_the_bits_of_a_whole_one(n_q, n_kv, d_head, window, dtype):
    t, kdim, T = (torch.bfloat16, torch.float16)[dtype], n_kv * d_head, 5000
    desc = kvd.make_desc(1, 256, n_q, n_kv, d_head, 1e-6, False, 1e-6, 0, 1, T + 64, 1)
    c = kvd.Kvd(desc)
    c.kvd_set_dtype(dtype)
    g = torch.Generator(device="cuda").manual_seed(d_head + n_q + window)
    c.kvd_set_layer(0, (torch.randn((256, 2 * kdim), generator=g, device="cuda") * 0.02).to(t), torch.ones(256, device="cuda").to(t), None, 1e4, window)
    c.kvd_attach_workspace(torch.empty(kvd.kvd_workspace_bytes(desc), dtype=torch.uint8, device="cuda"))
    k, v = (torch.randn((T, kdim), generator=g, device="cuda").to(t) for _ in range(2))
    q = torch.randn((2 * T, n_q, d_head), generator=g, device="cuda").to(t)
    k *= torch.linspace(0.2, 3.0, T, device="cuda").to(t)[:, None]
    group = n_q // n_kv
    for keys in [64 * n for n in range(6, 14)] + [T]:
        cut = keys // 2 + 13
        segs = [(k, v, kdim, 3, cut), (k[cut:], v[cut:], kdim, cut + 20, keys - cut - 21)]  # positions 3 .., a gap of 17
        n = min(60, 74 // n_kv * (128 // group))  # rows of the short call: at most 74 tiles
        whole = 128 // group * (148 // n_kv + 1)   # rows of the long one
        pos = torch.arange(keys - n, keys, dtype=torch.int32, device="cuda")
        pos[1] = 1  # sees no key
        long_pos = torch.cat((pos, torch.randint(3, keys, (whole - n,), generator=g, device="cuda").to(torch.int32)))
        ref = torch.zeros_like(q[:whole])
        c.kvd_prefill_attention(0, whole, q, long_pos, segs, 0.0, ref)
        for rows in {n, 1, min(n, 37)}:
            out = torch.full_like(q[:n + 1], 9.0)
            c.kvd_prefill_attention(0, rows, q, pos, segs, 0.0, out)
            assert torch.equal(out[:rows], ref[:rows]) and bool((out[rows:] == 9).all()), (keys, rows)
        assert bool((ref[1] == 0).all()) and bool(torch.isfinite(ref.float()).all())
    # as many tiles as are shared, each with a walk of its own: from no block (rows in front of the first key) and one to all
    for keys, first in ((700, 3), (T - 20, 3)):
        n = 74 // n_kv * (128 // group) - 3
        segs = [(k, v, kdim, first, keys // 2), (k[keys // 2:], v[keys // 2:], kdim, first + keys // 2 + 17, keys - keys // 2)]
        pos = (torch.arange(n, device="cuda") * (keys + 25) // n).to(torch.int32)
        more = torch.full((128 // group * (148 // n_kv + 1) - n,), keys, dtype=torch.int32, device="cuda")
        ref, out = torch.zeros_like(q[:n + len(more)]), torch.full_like(q[:n + 1], 9.0)
        c.kvd_prefill_attention(0, n + len(more), q, torch.cat((pos, more)), segs, 0.0, ref)
        c.kvd_prefill_attention(0, n, q, pos, segs, 0.0, out)
        assert torch.equal(out[:n], ref[:n]) and bool((out[n] == 9).all()) and bool((out[0] == 0).all()), keys
    assert c.kvd_poll_status() == kvd.KVD_OK
    c.close()
