"""Decode attention where its streaming kernels' ways of fetching keys change: the tensor-core kernel's ring of three and of
four pieces per warp (grids around three CTAs per SM), chunks of two and of more iterations, runs of keys that cross the edges
of segments, of the window and of the query's position; and the merge kernel's CTAs of one query head and of a whole group.

The reference is softmax attention in 64 bits on the same inputs; tolerance of the other attention tests (1e-2 of the norm and
of the largest value: 16-bit outputs and, in the tensor-core kernel, 16-bit weights)."""
import math

import pytest
import torch

import paper_2603_19664_b200 as kvd

pytestmark = pytest.mark.gpu

# query heads, KV heads, d_head: groups of 4 and 3 (tensor cores) and of 2 (fp32), every head size
LAYERS = {"g4-128": (16, 4, 128), "g3-64": (9, 3, 64), "g8-128": (8, 1, 128), "g4-64": (8, 2, 64), "g2-256": (8, 4, 256), "g2-128": (4, 2, 128)}


def _reference(q, k, v, pos, q_pos, window):
    seen = (pos <= q_pos) & ((q_pos - pos < window) if window else True)
    group = q.shape[0] // k.shape[1]
    k, v = (t[seen].double().repeat_interleave(group, 1) for t in (k, v))
    score = torch.einsum("hd,nhd->hn", q.double(), k) / math.sqrt(q.shape[-1])
    return torch.einsum("hn,nhd->hd", score.softmax(-1), v)


@pytest.mark.parametrize("half", [False, True], ids=["bf16", "f16"])
@pytest.mark.parametrize("layer", LAYERS)
@pytest.mark.parametrize("batch,ctx,cuts,window", [
    (1, 37, (), 0),                    # less than one iteration
    (1, 700, (1, 333, 699), 0),        # four segments, edges inside runs of keys
    (2, 1501, (1500,), 0),             # the new token by itself
    (3, 2000, (1000, 1744), 517),      # a window that starts inside a run
    (9, 1300, (1299,), 0), (13, 1300, (17,), 0),  # grids on both sides of three CTAs per SM
    (1, 9001, (4500,), 0),             # chunks of more than two iterations (every piece of the ring used again)
    (33, 900, (899,), 0),              # merge CTAs of a whole group
])
def test_keys_however_they_are_fetched(layer, half, batch, ctx, cuts, window):
    nq, nkv, dh = LAYERS[layer]
    dt, kdim = torch.float16 if half else torch.bfloat16, nkv * dh
    desc = kvd.make_desc(1, 64, nq, nkv, dh, 1e-6, False, 1e-6, kvd.KVD_ROPE_INTERLEAVED, 1, ctx + 64, batch)
    c = kvd.Kvd(desc)
    if half:
        c.kvd_set_dtype(1)
    g = torch.Generator(device="cuda").manual_seed(batch * ctx)
    draw = lambda *shape: torch.randn(shape, generator=g, device="cuda").to(dt)  # noqa: E731
    c.kvd_set_layer(0, draw(64, 2 * kdim), draw(64), None, 1e4, window)
    c.kvd_attach_workspace(torch.empty(kvd.kvd_workspace_bytes(desc), dtype=torch.uint8, device="cuda"))
    lens = [max(1, ctx - 5 * b) for b in range(batch)]
    q, out = draw(batch, nq, dh), torch.zeros((batch, nq, dh), dtype=dt, device="cuda")
    k, v = draw(batch, ctx, nkv, dh), draw(batch, ctx, nkv, dh)
    segs = []
    for b, n in enumerate(lens):
        edges = [0] + [x for x in cuts if x < n] + [n]
        segs.append([(k[b, i], v[b, i], kdim, i, j - i) for i, j in zip(edges, edges[1:])])
    q_pos = [n - 1 - b % 2 for b, n in enumerate(lens)]  # (every other query does not see the last key)
    c.kvd_decode_attention(0, batch, q, q_pos, segs, 0.0, out)
    assert c.kvd_poll_status() == kvd.KVD_OK
    for b, n in enumerate(lens):
        if q_pos[b] < 0:
            assert not out[b].any()
            continue
        want = _reference(q[b], k[b, :n], v[b, :n], torch.arange(n, device="cuda"), q_pos[b], window)
        err = (out[b].double() - want).abs()
        assert err.norm() <= 1e-2 * want.norm() and err.max() <= 1e-2 * want.abs().max(), b
    c.close()
