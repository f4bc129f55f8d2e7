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
LAYERS = {"g4-128": (16, 4, 128), "g4-128-8": (32, 8, 128), "g3-64": (9, 3, 64), "g8-128": (8, 1, 128), "g4-64": (8, 2, 64), "g2-256": (8, 4, 256), "g2-128": (4, 2, 128)}


def _reference(q, k, v, pos, q_pos, window):
    seen = (pos <= q_pos) & ((q_pos - pos < window) if window else True)
    group = q.shape[0] // k.shape[1]
    k, v = (t[seen].double().repeat_interleave(group, 1) for t in (k, v))
    score = torch.einsum("hd,nhd->hn", q.double(), k) / math.sqrt(q.shape[-1])
    return torch.einsum("hn,nhd->hd", score.softmax(-1), v)


CASES = [  # batch, ctx, cuts, window
    (1, 37, (), 0),                    # less than one iteration
    (1, 700, (1, 333, 699), 0),        # four segments, edges inside runs of keys
    (2, 1501, (1500,), 0),             # the new token by itself
    (3, 2000, (1000, 1744), 517),      # a window that starts inside a run
    (9, 1300, (1299,), 0), (13, 1300, (17,), 0), (64, 1100, (1000,), 0),  # grids on both sides of three CTAs per SM, merge CTAs of a whole group
    (1, 9001, (4500,), 0), (33, 900, (899,), 0),
    (1, 10000, (9999,), 0), (1, 14000, (7001,), 0), (1, 20001, (300,), 0),  # chunks of more than two iterations: pieces of the ring used again
]


def _lengths(batch, ctx):
    """Keys of each sequence and its query's position (every other query does not see the last key)."""
    lens = [max(2, ctx - 5 * b) for b in range(batch)]
    return lens, [n - 1 - b % 2 for b, n in enumerate(lens)]


def _regime(layer, batch, ctx, window, sms):
    """(pieces per warp, iterations per chunk, a merge CTA takes a whole group) of a launch, by the rules of the launch."""
    nq, nkv, dh = LAYERS[layer]
    splits = [kvd.binding.kvd_attention_split(dh, nkv, max(0, q - window + 1) if window else 0, q) for q in _lengths(batch, ctx)[1]]
    iters = max(keys for _, keys in splits) // (32 // (dh // 8) * 8 * 4)
    group = max(1, 16 // (nq // nkv))
    warps = min(20, -(-max(n for n, _ in splits) // group))
    return 4 if sum(n for n, _ in splits) * nkv <= 3 * sms else 3, iters, batch * nq * (dh // 64) * warps > 20 * sms


def test_the_cases_reach_both_rings_long_chunks_and_both_merges():
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    reached = {layer: [_regime(layer, b, ctx, w, sms) for b, ctx, _, w in CASES] for layer in LAYERS}
    for layer, (nq, nkv, dh) in LAYERS.items():
        if nq // nkv >= 3 and dh <= 128:
            assert {p for p, _, _ in reached[layer]} == {3, 4}, layer
    assert {(p, i > 2) for p, i, _ in reached["g4-128-8"]} == {(3, False), (3, True), (4, False), (4, True)}
    assert max(i for _, i, _ in reached["g4-128-8"]) >= 5 and max(i for _, i, _ in reached["g2-256"]) >= 3
    for layer in ("g4-128", "g4-128-8", "g8-128", "g2-256"):
        assert {m for _, _, m in reached[layer]} == {False, True}, layer


@pytest.mark.parametrize("half", [False, True], ids=["bf16", "f16"])
@pytest.mark.parametrize("layer", LAYERS)
@pytest.mark.parametrize("batch,ctx,cuts,window", CASES)
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
    lens, q_pos = _lengths(batch, ctx)
    q, out = draw(batch, nq, dh), torch.zeros((batch, nq, dh), dtype=dt, device="cuda")
    k, v = draw(batch, ctx, nkv, dh), draw(batch, ctx, nkv, dh)
    segs = []
    for b, n in enumerate(lens):
        edges = [0] + [x for x in cuts if x < n] + [n]
        segs.append([(k[b, i], v[b, i], kdim, i, j - i) for i, j in zip(edges, edges[1:])])
    c.kvd_decode_attention(0, batch, q, q_pos, segs, 0.0, out)
    assert c.kvd_poll_status() == kvd.KVD_OK
    for b, n in enumerate(lens):
        want = _reference(q[b], k[b, :n], v[b, :n], torch.arange(n, device="cuda"), q_pos[b], window)
        err = (out[b].double() - want).abs()
        assert err.norm() <= 1e-2 * want.norm() and err.max() <= 1e-2 * want.abs().max(), b
    c.close()
