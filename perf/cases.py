"""What the framework's speed is measured on: one layer's calls of a decode step, a prefill segment and the
lower-precision checkpoints, and a whole decoder block, over the range of shapes, batch sizes and lengths that the
configurations, tests and benchmark of this repository use.

A case is a dict: ``kind`` (which calls a pass makes, see the ``_prepare_*`` functions), ``model`` (a layer shape of
``SHAPES``), ``dtype`` of rows, weights, K/V and outputs, and sizes:

  ctx     tokens of context behind the new ones    batch   sequences decoded together
  live    of these, the last ones whose K/V are kept (the others' are rebuilt from their rows)
  new     tokens of the segment (kind "turn")      layers  decoder blocks (kind "block")

Sequences of a batch are ragged (a few tokens shorter each), so no row count is a multiple of a tile.  The new rows of a
decode step are appended to a slot of the store that the pass empties first, so that a pass can be repeated; nothing
else of the state changes.
"""
import math

import torch

import paper_2603_19664_b200 as kvd

# d_hidden, query heads, KV heads, d_head, key norm, rotation base, sliding window, MLP width, vocabulary
SHAPES = {
    "smollm2-135m": dict(d=576, nq=9, nkv=3, dh=64, norm=False, theta=1.0e4, window=0, mlp=1536, vocab=49152),
    "gemma3-4b": dict(d=2560, nq=8, nkv=4, dh=256, norm=True, theta=1.0e6, window=0, mlp=10240, vocab=262144),
    "gemma3-4b-local": dict(d=2560, nq=8, nkv=4, dh=256, norm=True, theta=1.0e4, window=1024, mlp=10240, vocab=262144),
    "qwen3-4b": dict(d=2560, nq=32, nkv=8, dh=128, norm=True, theta=1.0e6, window=0, mlp=9728, vocab=151936),
}
DTYPES = {"bf16": (0, torch.bfloat16), "f16": (1, torch.float16), "f32": (2, torch.float32)}
EPS = 1e-6


def listed():
    return [
        # the smallest layer and context: launches and latency are all there is
        dict(name="smol_step_512", kind="step", model="smollm2-135m", dtype="bf16", ctx=512),
        # the benchmark's step: checkpoint 4096 rows, rebuild their K/V, attend over them
        dict(name="gemma_step_4096", kind="step", model="gemma3-4b", dtype="bf16", ctx=4096),
        # decode step of a global layer under the bounded cache: 2048 tokens of context, 256 of them live
        dict(name="gemma_decode_b4", kind="decode", model="gemma3-4b", dtype="bf16", batch=4, ctx=2048, live=256),
        # the largest decode batch on a sliding-window layer
        dict(name="gemma_local_decode_b64", kind="decode", model="gemma3-4b-local", dtype="bf16", batch=64, ctx=2048, live=256),
        # the same step with every K/V kept: the full-cache arm, in fp16
        dict(name="gemma_cached_b16_f16", kind="cached", model="gemma3-4b", dtype="f16", batch=16, ctx=2048),
        # one long sequence from the cache: the read that recomputation is compared with
        dict(name="gemma_cached_32768", kind="cached", model="gemma3-4b", dtype="bf16", batch=1, ctx=32768),
        # the long-context batch: 8 sequences of 32768 tokens, 512 live, everything else rebuilt (the largest case)
        dict(name="qwen_decode_32768_b8", kind="decode", model="qwen3-4b", dtype="bf16", batch=8, ctx=32768, live=512),
        # one turn of a conversation: a user's 837 tokens on top of 7013, of which 256 are live
        dict(name="gemma_turn_837", kind="turn", model="gemma3-4b", dtype="bf16", new=837, ctx=7013, live=256),
        # a prompt with nothing before it
        dict(name="qwen_prefill_4096", kind="turn", model="qwen3-4b", dtype="bf16", new=4096, ctx=0, live=0),
        # E4M3 checkpoints, rebuilt and attended in one kernel
        dict(name="gemma_fp8_4096", kind="fp8", model="gemma3-4b", dtype="bf16", batch=1, ctx=4096),
        # 4-bit checkpoints of a small ragged batch
        dict(name="gemma_fp4_1000_b3", kind="fp4", model="gemma3-4b", dtype="bf16", batch=3, ctx=1000),
        # one token through three whole decoder blocks and the vocabulary projection
        dict(name="gemma_block_b1", kind="block", model="gemma3-4b", dtype="bf16", layers=3, batch=1, ctx=2048),
    ]


def _log(rng, lo, hi):
    """A whole number spread over the logarithm of lo..hi."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["step", "decode", "decode", "cached", "cached", "turn", "turn", "fp8", "fp4", "block", "block"])
    big = rng.choice(["gemma3-4b", "gemma3-4b-local", "qwen3-4b"])
    if kind == "step":
        model = rng.choice(["smollm2-135m", "gemma3-4b", "qwen3-4b"])
        return dict(kind=kind, model=model, dtype=rng.choice(["bf16", "bf16", "bf16", "f16", "f32"]), ctx=_log(rng, 16, 32768))
    if kind == "decode":
        batch = _log(rng, 1, 64)
        ctx = _log(rng, 256, min(32768, 262144 // batch))
        return dict(kind=kind, model=big, dtype="bf16", batch=batch, ctx=ctx, live=_log(rng, 16, min(512, ctx - 128)))
    if kind == "cached":
        batch = _log(rng, 1, 64)
        return dict(kind=kind, model=rng.choice([big, "smollm2-135m"]), dtype=rng.choice(["bf16", "bf16", "f16"]), batch=batch,
                    ctx=_log(rng, 128, min(32768, 262144 // batch)))
    if kind == "turn":
        ctx = rng.choice([0, _log(rng, 512, 8192)])
        return dict(kind=kind, model=rng.choice([big, "smollm2-135m"]), dtype=rng.choice(["bf16", "bf16", "f16"]),
                    new=_log(rng, 16, 4096), ctx=ctx, live=256 if ctx else 0)
    if kind in ("fp8", "fp4"):
        batch = _log(rng, 1, 16)
        model = rng.choice(["gemma3-4b", "qwen3-4b"])
        return dict(kind=kind, model=model, dtype="bf16", batch=batch, ctx=_log(rng, 256, min(16384, 32768 // batch)))
    batch = _log(rng, 1, 64)
    return dict(kind=kind, model=rng.choice(["gemma3-4b", "gemma3-4b-local", "qwen3-4b"]), dtype="bf16", layers=rng.randint(1, 3),
                batch=batch, ctx=_log(rng, 256, min(8192, 131072 // batch)))


# ----------------------------------------------------------------------------------------------- what a program keeps
class _Draws:
    """The random inputs of one state, drawn in a fixed order from the seed."""

    def __init__(self, case, seed):
        self.case, self.s = case, SHAPES[case["model"]]
        self.code, self.dt = DTYPES[case["dtype"]]
        self.kdim = self.s["nkv"] * self.s["dh"]
        self.g = torch.Generator(device="cuda")
        self.g.manual_seed(seed)
        # residual rows are N(0, 1) with one channel in a hundred twenty times larger, as real residual streams have them
        self.gain = torch.ones(self.s["d"], device="cuda")
        self.gain[torch.randperm(self.s["d"], generator=self.g, device="cuda")[: self.s["d"] // 100]] = 20.0

    def normal(self, shape, std=1.0, mean=0.0):
        return torch.randn(shape, generator=self.g, device="cuda").mul_(std).add_(mean).to(self.dt)

    def rows(self, n):
        return torch.randn((n, self.s["d"]), generator=self.g, device="cuda").mul_(self.gain).to(self.dt)

    def layer(self):
        """Norm scale of the input, norm scale of the keys (or None), K and V projection of a layer."""
        s = self.s
        gamma_in = self.normal((s["d"],), 0.02, 1.0)
        gamma_k = self.normal((s["dh"],), 0.02, 1.0) if s["norm"] else None
        return gamma_in, gamma_k, self.normal((s["d"], 2 * self.kdim), 0.02)

    def lo(self, pos):
        """First position that a query at `pos` sees."""
        return max(0, pos - self.s["window"] + 1) if self.s["window"] else 0


class _State(_Draws):
    """A context, the buffers of its calls, and the inputs of one pass."""

    def __init__(self, case, seed, max_seqs, max_tokens, max_batch, layers=1):
        super().__init__(case, seed)
        s = self.s
        self.desc = kvd.make_desc(layers, s["d"], s["nq"], s["nkv"], s["dh"], EPS, s["norm"], EPS, kvd.KVD_ROPE_INTERLEAVED,
                                  max_seqs, max_tokens, max_batch)
        self.ctx = kvd.Kvd(self.desc)
        if self.code:
            self.ctx.kvd_set_dtype(self.code)
        self.gamma_in = []
        for layer in range(layers):
            gamma_in, gamma_k, w = self.layer()
            self.gamma_in.append(gamma_in)
            self.ctx.kvd_set_layer(layer, w, gamma_in, gamma_k, s["theta"], s["window"])
        self.ws = torch.empty(kvd.kvd_workspace_bytes(self.desc), dtype=torch.uint8, device="cuda")
        self.ctx.kvd_attach_workspace(self.ws)

    def kv(self, *shape):
        return (torch.zeros((*shape, self.kdim), dtype=self.dt, device="cuda"), torch.zeros((*shape, self.kdim), dtype=self.dt, device="cuda"))

    def store(self, layers=1):
        self.arena = torch.zeros(kvd.kvd_store_bytes_dtype(self.desc, layers, self.code), dtype=torch.uint8, device="cuda")
        self.ctx.kvd_attach_store(self.arena, layers)

    def query(self, n):
        self.q = self.normal((n, self.s["nq"], self.s["dh"]))
        self.out = torch.zeros_like(self.q)


def _ints(values):
    return torch.tensor(list(values), dtype=torch.int32, device="cuda")


def _lengths(case):
    """Context length of each sequence of a batch."""
    return [max(1, case["ctx"] - 3 * b) for b in range(case["batch"])]


# ---- kind "step": STORE_RESIDUAL of a context, its K/V from the store with the new token's in the same launch, attention
def _prepare_step(case, seed):
    n = case["ctx"]
    st = _State(case, seed, 1, n + 1, 1)
    st.store()
    st.x, st.pos = st.rows(n + 1), _ints(range(n + 1))
    st.k, st.v = st.kv(n + 1)
    st.query(1)
    st.stored = st.arena[: n * st.s["d"] * st.x.element_size()].view(st.dt).view(n, st.s["d"])
    return st


def _run_step(st):
    n, c = st.case["ctx"], st.ctx
    c.kvd_reset_sequence(0)
    c.kvd_checkpoint_residual(0, 0, st.x, st.pos, n)
    c.kvd_recompute_kv_step(0, [(0, 0, n, st.k, st.v)], st.x[n:], st.pos[n:], 1, st.k[n:], st.v[n:], st.kdim)
    if st.code == 2:  # attention has no fp32 form
        return st.stored, st.k, st.v
    c.kvd_decode_attention(0, 1, st.q, [n], [[(st.k, st.v, st.kdim, 0, n), (st.k[n:], st.v[n:], st.kdim, n, 1)]], 0.0, st.out)
    return st.stored, st.k, st.v, st.out


# ---- kind "decode": one token per sequence, K/V of evicted positions rebuilt, `live` positions kept
def _prepare_decode(case, seed):
    b_, live, lens = case["batch"], case["live"], _lengths(case)
    st = _State(case, seed, b_ + 1, max(max(lens) + 1, b_), b_)
    st.store()
    pos = _ints(range(max(lens)))
    for b, n in enumerate(lens):
        st.ctx.kvd_checkpoint_residual(b, 0, st.rows(n), pos, n)
    st.lens, st.x, st.pos = lens, st.rows(b_), _ints(lens)
    lo = [st.lo(n) for n in lens]
    keep = [min(live, n - a) for n, a in zip(lens, lo)]
    first = [n - k for n, k in zip(lens, keep)]  # first live position
    st.n_old = [max(0, f - a) for f, a in zip(first, lo)]
    st.old_k, st.old_v = st.kv(b_, max(1, max(st.n_old)))
    st.live_k, st.live_v = st.kv(b_, live + 1)
    for b in range(b_):  # the new token's place is the last one: the window ends right before it
        at = live - keep[b]
        if keep[b]:
            st.ctx.kvd_recompute_kv(0, None, None, keep[b], st.live_k[b, at], st.live_v[b, at], st.kdim, seq=b, first_row=first[b])
    st.ranges = [(b, lo[b], st.n_old[b], st.old_k[b], st.old_v[b]) for b in range(b_) if st.n_old[b]]
    st.segs = []
    for b in range(b_):
        at = live - keep[b]
        one = [(st.old_k[b], st.old_v[b], st.kdim, lo[b], st.n_old[b])] if st.n_old[b] else []
        st.segs.append(one + [(st.live_k[b, at], st.live_v[b, at], st.kdim, first[b], keep[b] + 1)])
    st.slots = [b_] * b_
    st.query(b_)
    return st


def _run_decode(st):
    b_, live, c = st.case["batch"], st.case["live"], st.ctx
    c.kvd_reset_sequence(b_)
    c.kvd_decode_step_kv(0, st.ranges, st.kdim, st.x, st.pos, b_, st.slots, st.live_k[:, live], st.live_v[:, live], (live + 1) * st.kdim)
    c.kvd_decode_attention(0, b_, st.q, st.lens, st.segs, 0.0, st.out)
    return st.old_k, st.old_v, st.live_k, st.live_v, st.out


# ---- kind "cached": one token per sequence, every K/V kept
def _prepare_cached(case, seed):
    b_, lens = case["batch"], _lengths(case)
    st = _State(case, seed, 1, max(max(lens) + 1, b_), b_)
    st.store()
    st.lens, st.x, st.pos = lens, st.rows(b_), _ints(lens)
    room = case["ctx"] + 1  # position p of sequence b lies where the new tokens share a column of the buffer
    st.k, st.v = st.normal((b_, room, st.kdim)), st.normal((b_, room, st.kdim))
    st.segs = []
    for b, n in enumerate(lens):
        a = st.lo(n)
        at = room - 1 - n + a
        st.segs.append([(st.k[b, at], st.v[b, at], st.kdim, a, n + 1 - a)])
    st.slots = [0] * b_
    st.query(b_)
    return st


def _run_cached(st):
    b_, c, n = st.case["batch"], st.ctx, st.case["ctx"]
    c.kvd_reset_sequence(0)
    c.kvd_decode_step_kv(0, [], st.kdim, st.x, st.pos, b_, st.slots, st.k[:, n], st.v[:, n], (n + 1) * st.kdim)
    c.kvd_decode_attention(0, b_, st.q, st.lens, st.segs, 0.0, st.out)
    return st.k[:, n], st.v[:, n], st.out


# ---- kind "turn": a segment of new tokens of one sequence, on top of `ctx` tokens of which `live` have kept K/V
def _prepare_turn(case, seed):
    new, ctx, live = case["new"], case["ctx"], case["live"]
    st = _State(case, seed, 2, ctx + new, 1)
    st.store()
    if ctx:
        st.ctx.kvd_checkpoint_residual(0, 0, st.rows(ctx), _ints(range(ctx)), ctx)
    st.x, st.pos = st.rows(new), _ints(range(ctx, ctx + new))
    st.k, st.v = st.kv(live + new)
    st.lo_min = st.lo(ctx)
    st.n_old = max(0, ctx - live - st.lo_min)
    st.old_k, st.old_v = st.kv(max(1, st.n_old))
    st.first = ctx - live
    if live:
        st.ctx.kvd_recompute_kv(0, None, None, live, st.k, st.v, st.kdim, seq=0, first_row=st.first)
    st.segs = ([(st.old_k, st.old_v, st.kdim, st.lo_min, st.n_old)] if st.n_old else []) + [(st.k, st.v, st.kdim, st.first, live + new)]
    st.query(new)
    return st


def _run_turn(st):
    new, live, c = st.case["new"], st.case["live"], st.ctx
    c.kvd_reset_sequence(1)
    c.kvd_checkpoint_residual(1, 0, st.x, st.pos, new)
    c.kvd_recompute_kv(0, st.x, st.pos, new, st.k[live:], st.v[live:], st.kdim)
    if st.n_old:
        c.kvd_recompute_kv(0, None, None, st.n_old, st.old_k, st.old_v, st.kdim, seq=0, first_row=st.lo_min)
    c.kvd_prefill_attention(0, new, st.q, st.pos, st.segs, 0.0, st.out)
    return st.old_k, st.old_v, st.k, st.v, st.out


# ---- kind "fp8": E4M3 checkpoints rebuilt inside attention; the new tokens quantised, their K/V written
def _prepare_fp8(case, seed):
    b_, lens = case["batch"], _lengths(case)
    st = _State(case, seed, b_, max(lens) + 1, b_)
    st.arena = torch.zeros(kvd.kvd_store_bytes_fp8(st.desc, 1), dtype=torch.uint8, device="cuda")
    st.ctx.kvd_attach_store_fp8(st.arena, 1)
    pos = _ints(range(max(lens)))
    for b, n in enumerate(lens):
        st.ctx.kvd_checkpoint_residual_fp8(b, 0, st.rows(n), pos, n)
    st.lens, st.x, st.pos = lens, st.rows(b_), _ints(lens)
    st.codes = torch.zeros((b_, st.s["d"]), dtype=torch.uint8, device="cuda")
    st.scales, st.sumsq = torch.zeros(b_, device="cuda"), torch.zeros(b_, device="cuda")
    st.k, st.v = st.kv(b_)
    st.ranges = [(b, 0, n) for b, n in enumerate(lens)]
    st.segs = [[(st.k[b], st.v[b], st.kdim, n, 1)] for b, n in enumerate(lens)]
    st.query(b_)
    return st


def _run_fp8(st):
    b_, c = st.case["batch"], st.ctx
    c.kvd_quantize_rows_fp8(st.x, b_, st.codes, st.scales, st.sumsq)
    c.kvd_decode_attention_recompute_fp8_rows(0, b_, st.q, st.lens, st.ranges, [], (st.codes, st.scales, st.sumsq, st.pos, b_, st.k, st.v),
                                              st.kdim, st.segs, 0.0, st.out)
    return st.k, st.v, st.out


# ---- kind "fp4": 4-bit checkpoints, K/V rebuilt into a buffer, attention over it
def _prepare_fp4(case, seed):
    b_, lens = case["batch"], _lengths(case)
    st = _State(case, seed, b_, max(lens) + 1, b_)
    st.arena = torch.zeros(kvd.kvd_store_bytes_fp4(st.desc, 1), dtype=torch.uint8, device="cuda")
    st.ctx.kvd_attach_store_fp4(st.arena, 1)
    pos = _ints(range(max(lens)))
    for b, n in enumerate(lens):
        st.ctx.kvd_checkpoint_residual_fp4(b, 0, st.rows(n), pos, n)
    st.lens = lens
    st.last = [n - 1 for n in lens]
    st.scratch = torch.zeros(kvd.kvd_fp4_scratch_bytes(st.desc, sum(lens)), dtype=torch.uint8, device="cuda")
    st.k, st.v = st.kv(b_, max(lens))
    st.ranges = [(b, 0, n, st.k[b], st.v[b]) for b, n in enumerate(lens)]
    st.segs = [[(st.k[b], st.v[b], st.kdim, 0, n)] for b, n in enumerate(lens)]
    st.query(b_)
    return st


def _run_fp4(st):
    st.ctx.kvd_recompute_kv_fp4(0, st.ranges, st.kdim, st.scratch)
    st.ctx.kvd_decode_attention(0, st.case["batch"], st.q, st.last, st.segs, 0.0, st.out)
    return st.k, st.v, st.out


# ---- kind "block": one token per sequence through whole decoder blocks and the vocabulary projection (full cache)
def _prepare_block(case, seed):
    b_, layers, lens = case["batch"], case["layers"], _lengths(case)
    st = _State(case, seed, 1, max(max(lens) + 1, b_), b_, layers)
    s, c = st.s, st.ctx
    st.store(layers)
    d, width = s["d"], s["nq"] * s["dh"]
    st.lin, st.gamma_q, st.k, st.v, st.segs = [], [], [], [], []
    room = case["ctx"] + 1
    for layer in range(layers):
        st.gamma_q.append(st.normal((s["dh"],), 0.02, 1.0) if s["norm"] else None)
        st.lin.append((c.kvd_scaffold_linear_create(st.normal((d, width), 0.02), st.gamma_in[layer], d, width, EPS),
                       c.kvd_scaffold_linear_create(st.normal((width, d), 0.02), None, width, d),
                       c.kvd_scaffold_linear_create(st.normal((d, 2 * s["mlp"]), 0.02), st.normal((d,), 0.02, 1.0), d, 2 * s["mlp"], EPS),
                       c.kvd_scaffold_linear_create(st.normal((s["mlp"], d), 0.02), None, s["mlp"], d)))
        k, v = st.normal((b_, room, st.kdim)), st.normal((b_, room, st.kdim))
        st.k.append(k)
        st.v.append(v)
        segs = []
        for b, n in enumerate(lens):
            a = st.lo(n)
            at = room - 1 - n + a
            segs.append([(k[b, at], v[b, at], st.kdim, a, n + 1 - a)])
        st.segs.append(segs)
    st.head = c.kvd_scaffold_linear_create(st.normal((d, s["vocab"]), 0.02), st.normal((d,), 0.02, 1.0), d, s["vocab"], EPS)
    st.table = st.normal((s["vocab"], d))
    st.tokens = torch.randint(s["vocab"], (b_,), generator=st.g, device="cuda").to(torch.int32)
    st.lens, st.pos, st.slots = lens, _ints(lens), [0] * b_

    def buf(cols):
        return torch.zeros((b_, cols), dtype=st.dt, device="cuda")

    st.h, st.inner, st.logits = buf(d), buf(s["mlp"]), buf(st.head.out_cols)
    st.raw, st.y, st.gu, st.y2 = (buf(lin.out_cols) for lin in st.lin[0])
    st.query(b_)
    return st


def _run_block(st):
    s, c, b_, n = st.s, st.ctx, st.case["batch"], st.case["ctx"]
    d, act = s["d"], 1 if st.case["model"].startswith("qwen") else 0
    c.kvd_reset_sequence(0)
    c.kvd_scaffold_embed(st.table, st.tokens, b_, d, s["vocab"], st.h)
    for layer, (q, o, gate_up, down) in enumerate(st.lin):
        c.kvd_scaffold_linear(q, st.h, b_, st.raw, q.out_cols)
        c.kvd_scaffold_query_finish(layer, st.raw, q.out_cols, st.pos, b_, st.gamma_q[layer], st.q)
        k, v = st.k[layer], st.v[layer]
        c.kvd_decode_step_kv(layer, [], st.kdim, st.h, st.pos, b_, st.slots, k[:, n], v[:, n], (n + 1) * st.kdim)
        c.kvd_decode_attention(layer, b_, st.q, st.lens, st.segs[layer], 0.0, st.out)
        c.kvd_scaffold_linear(o, st.out, b_, st.y, o.out_cols)
        c.kvd_scaffold_add_rows(st.h, st.y, o.out_cols, b_, d)
        c.kvd_scaffold_linear(gate_up, st.h, b_, st.gu, gate_up.out_cols)
        c.kvd_scaffold_gated_act(st.gu, gate_up.out_cols, b_, s["mlp"], act, st.inner)
        c.kvd_scaffold_linear(down, st.inner, b_, st.y2, down.out_cols)
        c.kvd_scaffold_add_rows(st.h, st.y2, down.out_cols, b_, d)
    c.kvd_scaffold_linear(st.head, st.h, b_, st.logits, st.head.out_cols)
    return [st.h, st.logits] + [t[:, n] for t in st.k + st.v]


_KINDS = {"step": (_prepare_step, _run_step), "decode": (_prepare_decode, _run_decode), "cached": (_prepare_cached, _run_cached),
          "turn": (_prepare_turn, _run_turn), "fp8": (_prepare_fp8, _run_fp8), "fp4": (_prepare_fp4, _run_fp4),
          "block": (_prepare_block, _run_block)}


def prepare(case, seed):
    return _KINDS[case["kind"]][0](case, seed)


def run(state):
    return _KINDS[state.case["kind"]][1](state)


# --------------------------------------------------------------------------------------- what a pass cannot do without
def work(case):
    s, kind = SHAPES[case["model"]], case["kind"]
    es = 4 if case["dtype"] == "f32" else 2
    d, kdim, qdim, win = s["d"], s["nkv"] * s["dh"], s["nq"] * s["dh"], s["window"]
    project = 4.0 * d * kdim        # flops of one row's K and V
    pair = 4.0 * qdim               # flops of one query token with one key
    weights = 2.0 * d * kdim * es
    kv_row = 2.0 * kdim * es        # one token's K and V
    out = 2.0 * qdim * es           # one token's query and attention output

    def seen(n):  # keys that a query at position n sees, itself among them
        return min(n + 1, win) if win else n + 1

    if kind == "step":
        n = case["ctx"]
        flops = (n + 1) * project + (0 if es == 4 else (n + 1) * pair)
        return {"bytes": (2 * n + 1) * d * es + (n + 1) * kv_row + weights + out, "flops": flops}
    if kind == "turn":
        new, ctx, live = case["new"], case["ctx"], case["live"]
        lo = max(0, ctx - win + 1) if win else 0
        old = max(0, ctx - live - lo)
        keys = sum(seen(ctx + i) for i in range(new))
        return {"bytes": (2 * new + old) * d * es + (live + new + old) * kv_row + weights + new * out,
                "flops": (new + old) * project + keys * pair}
    b_, lens = case["batch"], _lengths(case)
    keys = sum(seen(n) for n in lens)
    if kind == "decode":
        live = sum(min(case["live"], seen(n) - 1) for n in lens)
        old = keys - b_ - live
        return {"bytes": (old + 2 * b_) * d * es + keys * kv_row + weights + b_ * out, "flops": (old + b_) * project + keys * pair}
    if kind == "cached":
        return {"bytes": 2 * b_ * d * es + keys * kv_row + weights + b_ * out, "flops": b_ * project + keys * pair}
    if kind == "fp8":
        return {"bytes": (keys - b_) * (d + 12.0) + b_ * (3 * d + kv_row + out) + weights / 2, "flops": keys * (project + pair)}
    if kind == "fp4":
        return {"bytes": (keys - b_) * (d / 2 + d / 16 + 12.0 + kv_row) + weights + b_ * out, "flops": (keys - b_) * (project + pair)}
    dense = 2.0 * d * qdim + 3.0 * d * s["mlp"]
    layer_bytes = weights + dense * es + keys * kv_row + b_ * d * es
    return {"bytes": case["layers"] * layer_bytes + d * s["vocab"] * es + b_ * (2 * d + s["vocab"]) * es,
            "flops": case["layers"] * (b_ * (project + 2 * dense) + keys * pair) + 2.0 * b_ * d * s["vocab"]}


def tolerance(case):
    """Four times what the outputs differ by from the same computation in 64 bits (``max`` is larger where the first
    tokens of a prompt attend to a few keys, and where errors pass through whole blocks)."""
    if case["kind"] == "block":  # 8e-3 and 3.8e-2 at three blocks
        return {"rel": 0.03, "max": 0.15}
    if case["dtype"] == "f32":   # TF32 products: 7.7e-4 and 2.2e-3
        return {"rel": 0.003, "max": 0.009}
    turn = case["kind"] == "turn"
    if case["dtype"] == "f16":   # 4e-4 and 1.6e-3 (7.4e-3)
        return {"rel": 0.0016, "max": 0.03 if turn else 0.0064}
    # 2.2e-3 to 3.2e-3, and 1.2e-2 (7.9e-2)
    return {"rel": 0.012, "max": 0.32 if turn else 0.05}


# ------------------------------------------------------------------------------------- the same outputs in 64 bits
def _normed(x, gamma):
    x = x.double()
    return x * (x.square().mean(-1, keepdim=True) + EPS).rsqrt() * gamma.double()


def _rotate(x, pos, theta):
    """Rotation of the pairs (2i, 2i + 1) of x [n, heads, d_head] by pos [n]."""
    dh = x.shape[-1]
    freq = theta ** (-torch.arange(0, dh, 2, dtype=torch.float64, device=x.device) / dh)
    angle = (pos.double()[:, None] * freq)[:, None, :]
    a, b, cos, sin = x[..., 0::2], x[..., 1::2], angle.cos(), angle.sin()
    return torch.stack((a * cos - b * sin, a * sin + b * cos), -1).flatten(-2)


def _heads(x, pos, gamma, theta, dh):
    """Head norm (where there is one) and rotation of [n, heads * d_head]."""
    x = x.view(x.shape[0], -1, dh)
    return _rotate(_normed(x, gamma) if gamma is not None else x, pos, theta).flatten(1)


def _project(dr, layer, x, pos, normed=None, w=None):
    """K and V [n, kdim] of rows x at positions pos (tensor)."""
    gamma_in, gamma_k, weight = layer
    w = weight.double() if w is None else w
    y = torch.cat([(_normed(x[i : i + 8192], gamma_in) if normed is None else normed[i : i + 8192]) @ w for i in range(0, x.shape[0], 8192)])
    return _heads(y[:, : dr.kdim].contiguous(), pos, gamma_k, dr.s["theta"], dr.s["dh"]), y[:, dr.kdim :].contiguous()


def _attend(dr, q, q_pos, k, v, first):
    """Attention of q [n, nq, dh] at positions q_pos over k, v [m, kdim] at positions first, first + 1, ..."""
    s = dr.s
    key = first + torch.arange(k.shape[0], device="cuda")
    seen = (key[None, :] <= q_pos[:, None]) & ((q_pos[:, None] - key[None, :] < s["window"]) if s["window"] else True)
    k, v = k.view(-1, s["nkv"], s["dh"]), v.view(-1, s["nkv"], s["dh"])
    group, out = s["nq"] // s["nkv"], torch.empty(q.shape, dtype=torch.float64, device="cuda")
    for h in range(s["nq"]):
        score = (q[:, h].double() @ k[:, h // group].T) / math.sqrt(s["dh"])
        out[:, h] = score.masked_fill_(~seen, -math.inf).softmax(-1) @ v[:, h // group]
    return out


def _arange(a, b):
    return torch.arange(a, b, device="cuda")


def _exact_step(case, seed):
    dr, n = _Draws(case, seed), case["ctx"]
    layer = dr.layer()
    x = dr.rows(n + 1)
    q = dr.normal((1, dr.s["nq"], dr.s["dh"]))
    k, v = _project(dr, layer, x, _arange(0, n + 1))
    if dr.code == 2:
        return x[:n].double(), k, v
    return x[:n].double(), k, v, _attend(dr, q, _arange(n, n + 1), k, v, 0)


def _exact_decode(case, seed):
    dr, b_, live, lens = _Draws(case, seed), case["batch"], case["live"], _lengths(case)
    layer = dr.layer()
    rows = [dr.rows(n) for n in lens]
    x = dr.rows(b_)
    q = dr.normal((b_, dr.s["nq"], dr.s["dh"]))
    lo = [dr.lo(n) for n in lens]
    keep = [min(live, n - a) for n, a in zip(lens, lo)]
    n_old = [n - p - a for n, p, a in zip(lens, keep, lo)]
    zeros = lambda room: torch.zeros((b_, room, dr.kdim), dtype=torch.float64, device="cuda")  # noqa: E731
    old_k, old_v, live_k, live_v = (zeros(room) for room in [max(1, max(n_old))] * 2 + [live + 1] * 2)
    out, w = torch.zeros(q.shape, dtype=torch.float64, device="cuda"), layer[2].double()
    for b, n in enumerate(lens):
        k, v = _project(dr, layer, torch.cat((rows[b][lo[b] :], x[b : b + 1])), _arange(lo[b], n + 1), w=w)
        rows[b] = None
        old_k[b, : n_old[b]], old_v[b, : n_old[b]] = k[: n_old[b]], v[: n_old[b]]
        live_k[b, live - keep[b] :], live_v[b, live - keep[b] :] = k[n_old[b] :], v[n_old[b] :]
        out[b] = _attend(dr, q[b : b + 1], _arange(n, n + 1), k, v, lo[b])[0]
    return old_k, old_v, live_k, live_v, out


def _exact_cached(case, seed):
    dr, b_, n, lens = _Draws(case, seed), case["batch"], case["ctx"], _lengths(case)
    layer = dr.layer()
    x = dr.rows(b_)
    k, v = dr.normal((b_, n + 1, dr.kdim)), dr.normal((b_, n + 1, dr.kdim))
    q = dr.normal((b_, dr.s["nq"], dr.s["dh"]))
    kn, vn = _project(dr, layer, x, _ints(lens))
    return kn, vn, _attend_cached(dr, q, lens, k, v, kn, vn)


def _attend_cached(dr, q, lens, k, v, kn, vn):
    """One query per sequence over its cache k, v [b, room, kdim], whose last column are the new tokens' kn, vn."""
    out = torch.empty(q.shape, dtype=torch.float64, device="cuda")
    for b, n in enumerate(lens):
        a = dr.lo(n)
        at = k.shape[1] - 1 - n + a
        kb, vb = (torch.cat((t[b, at:-1].double(), new[b : b + 1])) for t, new in ((k, kn), (v, vn)))
        out[b] = _attend(dr, q[b : b + 1], _arange(n, n + 1), kb, vb, a)[0]
    return out


def _exact_turn(case, seed):
    dr, new, ctx, live = _Draws(case, seed), case["new"], case["ctx"], case["live"]
    layer = dr.layer()
    rows = dr.rows(ctx) if ctx else None
    x = dr.rows(new)
    q = dr.normal((new, dr.s["nq"], dr.s["dh"]))
    lo = dr.lo(ctx)
    n_old = max(0, ctx - live - lo)
    start = min(lo, ctx - live)
    k, v = _project(dr, layer, torch.cat((rows[start:], x)) if ctx else x, _arange(start, ctx + new))
    out = _attend(dr, q, _arange(ctx, ctx + new), k, v, start)
    cut = ctx - live - start
    old = [t[lo - start : lo - start + n_old] if n_old else torch.zeros((1, dr.kdim), dtype=torch.float64, device="cuda") for t in (k, v)]
    return old[0], old[1], k[cut:], v[cut:], out


def _e4m3(x):
    return x.to(torch.float8_e4m3fn).float()


def _fp8_rows(x):
    """Rows as E4M3 codes and a scale decode (the statistic stays that of the row itself), over the row's rms."""
    x = x.float()
    amax = x.abs().amax(-1, keepdim=True).clamp_min(1e-30)
    decoded = _e4m3(x * (448.0 / amax)).double() * (amax / 448.0).double()
    return decoded * (x.double().square().mean(-1, keepdim=True) + EPS).rsqrt()


def _exact_fp8(case, seed):
    dr, b_, lens = _Draws(case, seed), case["batch"], _lengths(case)
    layer = dr.layer()
    rows = [dr.rows(n) for n in lens]
    x = dr.rows(b_)
    q = dr.normal((b_, dr.s["nq"], dr.s["dh"]))
    w = layer[0].float()[:, None] * layer[2].float()
    amax = w.abs().max()
    w = _e4m3(w * (448.0 / amax)).double() * (amax / 448.0).double()
    new_k, new_v, out = [], [], torch.empty(q.shape, dtype=torch.float64, device="cuda")
    for b, n in enumerate(lens):
        every = torch.cat((rows[b], x[b : b + 1]))
        k, v = _project(dr, layer, every, _arange(0, n + 1), _fp8_rows(every), w)
        new_k.append(k[n])
        new_v.append(v[n])
        out[b] = _attend(dr, q[b : b + 1], _arange(n, n + 1), k, v, 0)[0]
    return torch.stack(new_k), torch.stack(new_v), out


def _fp4_rows(x):
    """Rows as 4-bit codes under a scale of every 16 channels and one of the row decode, over the row's rms."""
    xf = x.float()
    _, ex = torch.frexp(xf.abs().amax(-1, keepdim=True))
    row = torch.exp2((ex - 11).double()).float()
    block = xf.view(x.shape[0], -1, 16)
    scale = _e4m3(block.abs().amax(-1) / 6.0 / row) * row
    quot = torch.where(scale[..., None] > 0, block / scale[..., None], torch.zeros_like(block))
    size = quot.abs()
    step = torch.where(size < 2, 0.5, torch.where(size < 4, 1.0, 2.0))
    code = (torch.round(size / step) * step).clamp_max(6.0) * quot.sign()
    decoded = (code * scale[..., None]).view(x.shape).double()
    return decoded * (x.double().square().mean(-1, keepdim=True) + EPS).rsqrt()


def _exact_fp4(case, seed):
    dr, b_, lens = _Draws(case, seed), case["batch"], _lengths(case)
    layer = dr.layer()
    rows = [dr.rows(n) for n in lens]
    q = dr.normal((b_, dr.s["nq"], dr.s["dh"]))
    k_out = torch.zeros((b_, max(lens), dr.kdim), dtype=torch.float64, device="cuda")
    v_out, out = torch.zeros_like(k_out), torch.empty(q.shape, dtype=torch.float64, device="cuda")
    for b, n in enumerate(lens):
        k, v = _project(dr, layer, rows[b], _arange(0, n), _fp4_rows(rows[b]) * layer[0].double())
        k_out[b, :n], v_out[b, :n] = k, v
        out[b] = _attend(dr, q[b : b + 1], _arange(n - 1, n), k, v, 0)[0]
    return k_out, v_out, out


def _exact_block(case, seed):
    dr, b_, n, lens = _Draws(case, seed), case["batch"], case["ctx"], _lengths(case)
    s = dr.s
    d, width, pos = s["d"], s["nq"] * s["dh"], _ints(lens)
    layers = [dr.layer() for _ in range(case["layers"])]
    rest = []
    for _ in layers:
        gamma_q = dr.normal((s["dh"],), 0.02, 1.0) if s["norm"] else None
        wq, wo = dr.normal((d, width), 0.02), dr.normal((width, d), 0.02)
        w1, gamma = dr.normal((d, 2 * s["mlp"]), 0.02), dr.normal((d,), 0.02, 1.0)
        w2 = dr.normal((s["mlp"], d), 0.02)
        rest.append((gamma_q, wq, wo, w1, gamma, w2, dr.normal((b_, n + 1, dr.kdim)), dr.normal((b_, n + 1, dr.kdim))))
    head, gamma_head = dr.normal((d, s["vocab"]), 0.02), dr.normal((d,), 0.02, 1.0)
    table = dr.normal((s["vocab"], d))
    h = table[torch.randint(s["vocab"], (b_,), generator=dr.g, device="cuda")].double()
    ks, vs = [], []
    for layer, (gamma_q, wq, wo, w1, gamma, w2, k, v) in zip(layers, rest):
        x = _normed(h, layer[0])
        q = _heads(x @ wq.double(), pos, gamma_q, s["theta"], s["dh"]).view(b_, s["nq"], s["dh"])
        kn, vn = _project(dr, layer, h, pos)
        h = h + _attend_cached(dr, q, lens, k, v, kn, vn).flatten(1) @ wo.double()
        gate, up = (_normed(h, gamma) @ w1.double()).chunk(2, -1)
        act = torch.nn.functional.silu(gate) if case["model"].startswith("qwen") else torch.nn.functional.gelu(gate, approximate="tanh")
        h = h + (act * up) @ w2.double()
        ks.append(kn)
        vs.append(vn)
    x = _normed(h, gamma_head)
    logits = torch.cat([x @ head[:, i : i + 32768].double() for i in range(0, s["vocab"], 32768)], -1)
    return [h, torch.nn.functional.pad(logits, (0, -s["vocab"] % 256))] + ks + vs  # columns up to a whole tile are zeros


_EXACT = {"step": _exact_step, "decode": _exact_decode, "cached": _exact_cached, "turn": _exact_turn, "fp8": _exact_fp8,
          "fp4": _exact_fp4, "block": _exact_block}


def exact(case, seed):
    return _EXACT[case["kind"]](case, seed)
