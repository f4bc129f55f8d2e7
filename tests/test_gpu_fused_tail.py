"""The fused recompute calls with a handful of live keys, which the merge kernel attends itself (at most 8 per sequence) instead
of a streaming launch: around that limit, ragged and mixed batches, gaps, windows that hide some or all of the recomputed keys,
keys that score minus infinity, and every head form of the fused kernel with both rotations.  Against the oracle or softmax
attention in 64 bits, with the tolerance of the other fused tests, and for the same bits alone and among others."""
import dataclasses
import math

import pytest
import torch

import paper_2603_19664_b200 as kvd
from kvd_synth import GEMMA3_4B_GLOBAL, GEMMA3_4B_LOCAL, QWEN3_4B
from test_gpu_fused import attn_check, run_case

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [GEMMA3_4B_GLOBAL, QWEN3_4B], ids=lambda s: s.name)
@pytest.mark.parametrize("n_old,n_live", [([300], 1), ([300], 6), ([300], 7), ([300], 8), ([1, 700, 0], 3), ([260] * 20, 2)])
def test_live_keys_around_what_the_merge_kernel_takes(shape, n_old, n_live):
    fused, two, ref = run_case(shape, n_old, n_live, seed=n_live)
    attn_check(fused, ref, "fused vs oracle")
    attn_check(fused, two, "fused vs two-call")


@pytest.mark.parametrize("window", [1, 2, 4, 5, 300])  # n_live + 1 = 4 live keys: some of them, all of them, with recomputed ones
def test_windows_over_the_live_keys(window):
    shape = dataclasses.replace(GEMMA3_4B_LOCAL, sliding_window=window)
    fused, two, ref = run_case(shape, [290, 513], 3, seed=window)
    attn_check(fused, ref, "fused vs oracle")
    attn_check(fused, two, "fused vs two-call")


class Step:
    """Fused steps over one small layer.  Sequence b: n_old[b] rows of the store at positions 0 .. n_old[b] - 1, live keys at
    n_old[b] + live[b][i] (ascending; a gap begins another segment), the query at the last of all.  kind: bf16, f16 or fp8."""
    D = 256

    def __init__(self, layer, n_old, live, kind="bf16", rope=kvd.KVD_ROPE_INTERLEAVED, seed=0):
        self.nq, self.nkv, self.dh = layer
        self.n_old, self.live, self.kind, self.kdim = n_old, live, kind, layer[1] * layer[2]
        self.dt, B = torch.float16 if kind == "f16" else torch.bfloat16, len(n_old)
        self.desc = kvd.make_desc(1, self.D, *layer, 1e-6, True, 1e-6, rope, B, max(n_old) + 64, B)
        self.c = kvd.Kvd(self.desc)
        if kind == "f16":
            self.c.kvd_set_dtype(1)
        g = torch.Generator(device="cuda").manual_seed(seed)
        draw = lambda *s: torch.randn(s, generator=g, device="cuda").to(self.dt)  # noqa: E731
        self.c.kvd_set_layer(0, draw(self.D, 2 * self.kdim) * self.D ** -0.5, 1 + 0.1 * draw(self.D), 1 + 0.1 * draw(self.dh), 1e4, 0)
        self.c.kvd_attach_workspace(torch.empty(kvd.kvd_workspace_bytes(self.desc), dtype=torch.uint8, device="cuda"))
        fp8 = kind == "fp8"
        arena = torch.empty((kvd.kvd_store_bytes_fp8 if fp8 else kvd.kvd_store_bytes)(self.desc, 1), dtype=torch.uint8, device="cuda")
        (self.c.kvd_attach_store_fp8 if fp8 else self.c.kvd_attach_store)(arena, 1)
        self.q, self.k, self.v = draw(B, self.nq, self.dh), [draw(len(p), self.nkv, self.dh) for p in live], [draw(len(p), self.nkv, self.dh) for p in live]
        self.rebuilt = []
        for b, n in enumerate(n_old):
            x, pos = draw(max(n, 1), self.D), torch.arange(max(n, 1), dtype=torch.int32, device="cuda")
            kb, vb = (torch.empty((n, self.nkv, self.dh), dtype=self.dt, device="cuda") for _ in range(2))
            if n:
                (self.c.kvd_checkpoint_residual_fp8 if fp8 else self.c.kvd_checkpoint_residual)(b, 0, x, pos, n)
                if fp8:
                    self.c.kvd_recompute_kv_fp8(0, [(b, 0, n, kb, vb)], self.kdim)
                else:
                    self.c.kvd_recompute_kv(0, None, None, n, kb, vb, self.kdim, seq=b, first_row=0)
            self.rebuilt.append((kb, vb))

    def run(self, seqs=None):
        """Output rows of a call over these sequences (all of them)."""
        seqs = list(range(len(self.n_old))) if seqs is None else seqs
        segs, q_pos = [], []
        for b in seqs:
            p, row = self.live[b], []
            for i in range(len(p)):
                if i == 0 or p[i] != p[i - 1] + 1:
                    row.append([self.k[b][i:], self.v[b][i:], self.kdim, self.n_old[b] + p[i], 0])
                row[-1][4] += 1
            segs.append([tuple(s) for s in row])
            q_pos.append(self.n_old[b] + p[-1] if p else max(self.n_old[b] - 1, 0))
        q, ranges = self.q[seqs].contiguous(), [(b, 0, self.n_old[b]) for b in seqs]
        out = torch.full_like(q, 9.0)
        if self.kind == "fp8":
            self.c.kvd_decode_attention_recompute_fp8(0, len(seqs), q, q_pos, ranges, [], self.kdim, segs, 0.0, out)
        else:
            self.c.kvd_decode_attention_recompute(0, len(seqs), q, q_pos, ranges, None, None, 0, None, None, self.kdim, segs, 0.0, out)
        assert self.c.kvd_poll_status() == kvd.KVD_OK
        return out

    def check(self, out):
        """Softmax attention in 64 bits over the keys and values that the library rebuilds (rounded to 16 bits) and the live
        ones; a key that scores minus infinity weighs nothing.  Tolerance of the other attention tests."""
        for b, row in enumerate(out):
            k, v = (torch.cat((a, l)).double().repeat_interleave(self.nq // self.nkv, 1) for a, l in zip(self.rebuilt[b], (self.k[b], self.v[b])))
            score = torch.einsum("hd,nhd->hn", self.q[b].double(), k) / math.sqrt(self.dh)
            weight = torch.exp(score - score.amax(1, keepdim=True).clamp(min=-1e30))
            total = weight.sum(1, keepdim=True)
            want = torch.einsum("hn,nhd->hd", weight / torch.where(total > 0, total, 1.0), v)
            err = (row.double() - want).abs()
            assert err.norm() <= 1e-2 * want.norm() and err.max() <= 1e-2 * want.abs().max(), b


GROUPS = {"2-256": (4, 2, 256), "1-256": (2, 2, 256), "4-128": (8, 2, 128), "2-128": (4, 2, 128), "1-128": (2, 2, 128)}  # all that the fused kernel exists for


@pytest.mark.parametrize("kind", ["bf16", "f16", "fp8"])
@pytest.mark.parametrize("layer", ["2-256", "4-128"])
@pytest.mark.parametrize("n_old,live,lost", [
    (300, [0], [0]), (300, [0, 1, 2], [0, 1, 2]), (300, [0, 1, 2], [1]), (700, list(range(8)), list(range(8))),
    (300, list(range(9)), list(range(9))), (0, [0, 1], [0, 1])])  # (nine: through the streaming kernel; none rebuilt: zeros)
def test_live_keys_that_score_minus_infinity(kind, layer, n_old, live, lost):
    """An overflowed key (16-bit stores of keys overflow to infinity) weighs nothing, also where it is the only live one."""
    s = Step(GROUPS[layer], [n_old], [live], kind)
    s.q[:, :, 5] = s.q[:, :, 5].abs() + 0.5
    for i in lost:
        s.k[0][i, 0, 5] = -math.inf  # for the first KV head's queries
    s.check(s.run())


@pytest.mark.parametrize("value", [math.nan, math.inf])
@pytest.mark.parametrize("kind", ["bf16", "f16"])
@pytest.mark.parametrize("layer", ["2-256", "4-128"])
@pytest.mark.parametrize("live", [[0], [0, 1, 2], list(range(9))])
def test_live_keys_that_score_nan_or_plus_infinity_give_what_the_two_calls_give(live, layer, kind, value):
    s = Step(GROUPS[layer], [300], [live], kind)
    s.q[:, :, 5] = s.q[:, :, 5].abs() + 0.5
    s.k[0][0, 0, 5] = value
    out, two = s.run(), torch.full_like(s.q, 9.0)
    segs = [(*s.rebuilt[0], s.kdim, 0, 300), (s.k[0], s.v[0], s.kdim, 300, len(live))]
    s.c.kvd_decode_attention(0, 1, s.q, [300 + live[-1]], [segs], 0.0, two)
    heads = s.nq // s.nkv  # of the first KV head
    assert torch.equal(out[:, :heads], two[:, :heads]) and s.c.kvd_poll_status() == kvd.KVD_OK
    attn_check(out[:, heads:].double().cpu().numpy(), two[:, heads:].double().cpu().numpy())


WIDE = {"2-256": (8, 4, 256), "4-128": (16, 4, 128)}  # (with 64 sequences more warps than the SMs hold at once: a merge CTA per KV head)
FEW, EIGHT, NINE = [0], list(range(8)), list(range(9))


@pytest.mark.parametrize("kind", ["bf16", "f16", "fp8"])
@pytest.mark.parametrize("layer", WIDE)
@pytest.mark.parametrize("n_old,live", [
    ([300, 300, 513], [FEW, NINE, EIGHT]),                                    # the streaming kernel takes the second one's
    ([20000, 300, 20300], [FEW, [], NINE]),                                   # more groups of partials than a merge CTA has warps
    ([260 + b for b in range(64)], [(FEW, EIGHT, NINE, [])[b % 4] for b in range(64)])], ids=["3", "long", "64"])
def test_a_sequence_gets_the_same_bits_alone_and_among_others(kind, layer, n_old, live):
    s = Step(WIDE[layer], n_old, live, kind)
    out = s.run()
    s.check(out)
    for b in range(min(len(n_old), 8)):
        assert torch.equal(s.run([b])[0], out[b]), b
        assert torch.equal(s.run([b, (b + 1) % len(n_old)])[0], out[b]), b
    before = s.c.kvd_launch_count()
    s.run([b for b, p in enumerate(live) if len(p) <= 8])
    assert s.c.kvd_launch_count() - before == 2  # (recompute, merge)
    before = s.c.kvd_launch_count()
    s.run()
    assert s.c.kvd_launch_count() - before == 3


@pytest.mark.parametrize("rope", [kvd.KVD_ROPE_INTERLEAVED, kvd.KVD_ROPE_HALF], ids=["pairs", "half-split"])
@pytest.mark.parametrize("kind", ["bf16", "f16", "fp8"])
@pytest.mark.parametrize("layer", GROUPS)
def test_every_head_form_with_both_rotations_and_gaps_between_live_keys(layer, kind, rope):
    s = Step(GROUPS[layer], [700, 300, 1, 513], [[0, 2, 3, 7], EIGHT, [4], [0, 1, 2, 5, 6, 7, 12, 13]], kind, rope, seed=3)
    s.check(s.run())


@pytest.mark.parametrize("kind", ["bf16", "f16", "fp8"])
@pytest.mark.parametrize("layer", WIDE)
@pytest.mark.parametrize("batch", [16, 64])  # a merge CTA per query head, per KV head
def test_batches_whose_live_keys_the_merge_kernel_takes(batch, layer, kind):
    s = Step(WIDE[layer], [260 + 3 * b for b in range(batch)], [list(range(1 + b % 8)) for b in range(batch)], kind, seed=batch)
    nq, _, dh = WIDE[layer]
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    assert (batch * nq * (dh // 64) * 2 > 20 * sms) == (batch == 64)  # (one warp for partials, one for live keys)
    before = s.c.kvd_launch_count()
    out = s.run()
    assert s.c.kvd_launch_count() - before == 2
    s.check(out)
