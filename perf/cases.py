"""The work that a user of this library has it do, as cases that can be timed one by one.

Three kinds of case, by the entry points that they call:

  projection  one multi-LoRA projection on one mixed batch: `mlora_mixed_forward`, with fine-tuning rows also
              `mlora_backward`, and `mlora_adamw_update` where the case trains
  set         the same over the seven projections of one decoder layer (q, k, v share an input, gate and up share one)
  layer       one whole decoder layer through `DecoderLayer`: `forward`, or `forward` and `backward` (which recomputes the
              layer for the fine-tuning rows from its saved input)

The rows of a batch are prompts, then decode rows (one token each), then rows of the base model alone, then fine-tuning
sequences.  Lengths are a function of the case; the adapters of prompts and decode rows, and every value, come from the seed.
Weights, buffers and, for the first two kinds, the plan are kept by the caller between calls, as a serving program keeps
them for the layers of a model; `DecoderLayer` makes a plan per call.  One context serves the whole process.
"""
from __future__ import annotations

import math
import weakref

import numpy as np
import torch

from paper_2607_28848_b200 import binding as mb
from paper_2607_28848_b200 import synth
from paper_2607_28848_b200.layer import DecoderLayer
from paper_2607_28848_b200.runner import Session, torch_dtype

RANKS = (8, 16, 32, 64, 128)
OWN_RANKS = (8, 16, 16, 32, 64, 128)        # ranks of the adapters of a layer that holds adapters of different ranks

_DEFAULTS = {"kind": "projection", "dtype": "bf16", "rank": 16, "adapters": 16, "zipf": False, "by_adapter": False,
             "own_ranks": False, "prompts": 0, "prompt_rows": 0, "decode_rows": 0, "base_rows": 0, "tune_rows": 0,
             "tune_seqs": 0, "tune_adapters": 0, "backward": False, "update": False, "dropout": 0.0}


def _case(name, **fields):
    c = dict(_DEFAULTS, **fields)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # The smallest call: a tiny fp32 layer (256 -> 256, four adapters of rank 8, 64 rows), forward and backward.
        _case("tiny_f32_step", d_in=256, d_out=256, dtype="f32", rank=8, adapters=4, prompts=3, prompt_rows=48,
              tune_rows=16, tune_seqs=1, tune_adapters=1, backward=True),
        # One decode step of a small server: 16 requests in flight, one projection.
        _case("decode16_q", d_in=4096, d_out=4096, adapters=4, decode_rows=16),
        # One decode step of 64 requests over all seven projections of a layer: every weight is read once for few rows.
        _case("decode64_set", kind="set", hidden=4096, kv=1024, ffn=14336, adapters=32, decode_rows=64),
        # A large decode batch over many adapters, rows in arrival order (5120 -> 13824, 128 adapters of rank 32).
        _case("decode512_r32", d_in=5120, d_out=13824, rank=32, adapters=128, decode_rows=512),
        # The fine-tuning step of a co-serving deployment: one adapter, a backward batch of 256 tokens, dropout 0.05, AdamW.
        _case("tune256_dropout_adamw", d_in=4096, d_out=4096, adapters=4, tune_rows=256, tune_seqs=2, tune_adapters=1,
              backward=True, update=True, dropout=0.05),
        # An ordinary mixed batch on one projection: 8 prompts, 64 decode rows, two fine-tuning sequences of 256 tokens.
        _case("mixed1600_q", d_in=4096, d_out=4096, prompts=8, prompt_rows=1024, decode_rows=64, tune_rows=512, tune_seqs=2,
              tune_adapters=2, backward=True),
        # Odd sizes: widths that fill no tile, a ragged batch with rows of the base model, rank 64.
        _case("ragged_r64", d_in=2880, d_out=7744, rank=64, adapters=8, prompts=5, prompt_rows=491, decode_rows=37,
              base_rows=29, tune_rows=301, tune_seqs=3, tune_adapters=2, backward=True),
        # Many adapters of different ranks (8 to 128) under Zipf popularity, rows ordered by adapter, half of them tuned.
        _case("ranks_8_to_128", d_in=4096, d_out=14336, rank=128, adapters=256, zipf=True, by_adapter=True, own_ranks=True,
              decode_rows=1024, tune_rows=1024, tune_seqs=4, tune_adapters=4, backward=True),
        # Decode rows beside one long fine-tuning sequence: the mix that co-serving is for.
        _case("decode512_tune2048_r32", d_in=5120, d_out=13824, rank=32, adapters=128, decode_rows=512, tune_rows=2048,
              tune_seqs=1, tune_adapters=1, backward=True),
        # A whole decoder layer serving prompts of up to a thousand tokens beside decode rows.
        _case("layer_serve", kind="layer", hidden=4096, heads=32, kv_heads=8, ffn=14336, adapters=32, prompts=3,
              prompt_rows=1920, decode_rows=128),
        # A whole decoder layer co-serving: mixed forward, then recompute and backward of four 512-token sequences.
        _case("layer_coserve", kind="layer", hidden=4096, heads=32, kv_heads=8, ffn=14336, adapters=32, prompts=6,
              prompt_rows=512, decode_rows=256, tune_rows=2048, tune_seqs=4, tune_adapters=4, backward=True),
        # The largest: 4096 mixed rows over the seven projections of a layer, forward and backward.
        _case("mixed4096_set", kind="set", hidden=4096, kv=1024, ffn=14336, adapters=32, prompts=12, prompt_rows=1024,
              decode_rows=1024, tune_rows=2048, tune_seqs=4, tune_adapters=4, backward=True),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same ranges: any mix of rows from one decode row up to 4096 rows, any rank, 1 to 256 adapters."""
    most = [max(work(c)[k] for c in listed()) for k in ("flops", "bytes")]
    while True:
        c = _draw(rng)
        w = work(c)
        if w["flops"] <= most[0] and w["bytes"] <= most[1]:
            return c


def _draw(rng):
    kind = rng.choice(("projection", "projection", "projection", "projection", "set", "layer"))
    c = _case(None, kind=kind, adapters=_log_uniform(rng, 1, 256), rank=rng.choice(RANKS))
    most = 4096
    if kind == "projection" and rng.random() < 0.1:       # fp32 layers are small
        c.update(dtype="f32", rank=rng.choice((4, 8, 16)), d_in=rng.randint(64, 512), d_out=rng.randint(64, 512),
                 adapters=_log_uniform(rng, 1, 16))
        most = 256
    elif kind == "projection":
        c.update(d_in=64 * _log_uniform(rng, 16, 224), d_out=64 * _log_uniform(rng, 16, 224))
    else:
        hidden = rng.choice((1024, 2048, 3072, 4096))
        c.update(hidden=hidden, ffn=64 * rng.randint(2 * hidden // 64, 7 * hidden // 128), adapters=min(c["adapters"], 64))
        if kind == "set":
            c.update(kv=hidden // rng.choice((1, 4)))
        else:                                             # heads of 128, in one layer of five of 64
            heads = hidden // (128 if rng.random() < 0.8 else 64)
            c.update(heads=heads, kv_heads=heads // rng.choice((1, 4)))
    use = rng.choice(("decode", "serve", "mixed", "mixed", "tune"))
    rows = _log_uniform(rng, 1 if use == "decode" else 33, min(most, 1024) if use == "decode" else most)
    if use == "decode":
        c.update(decode_rows=rows)
    elif use == "serve":
        d = rng.randint(0, rows // 3)
        c.update(prompts=rng.randint(1, 8), prompt_rows=rows - d, decode_rows=d)
    else:
        n = rng.randint(1, 4)
        t = rows if use == "tune" else rng.randint(rows // 4, rows // 2)
        left = rows - t
        d = rng.randint(0, left // 2)
        base = rng.randint(0, left // 16)
        c.update(tune_rows=t, tune_seqs=n, tune_adapters=min(rng.randint(1, n), c["adapters"]), decode_rows=d, base_rows=base,
                 prompts=rng.randint(1, 8) if left - d - base else 0, prompt_rows=left - d - base, backward=True)
        if kind == "projection" and use == "tune":
            c.update(dropout=rng.choice((0.0, 0.05)))
            if c["d_in"] % 4 == 0 and c["d_out"] % 4 == 0:
                c.update(update=rng.random() < 0.5)
    if c["decode_rows"]:
        c.update(zipf=rng.random() < 0.3, by_adapter=rng.random() < 0.3)
    if c["dtype"] == "bf16" and kind == "projection" and c["rank"] >= 32 and c["adapters"] > 1 and not c["dropout"]:
        c.update(own_ranks=rng.random() < 0.25)
    return c


# ---- the batch of a case --------------------------------------------------------------------------
def _lengths(total, parts):
    """`parts` lengths of unequal size with the given sum."""
    parts = min(parts, total)
    if parts < 1:
        return []
    cuts = [0] + [max(i, total * (2 * i + (i * 5) % 3) // (2 * parts + (parts * 5) % 3)) for i in range(1, parts)] + [total]
    return [b - a for a, b in zip(cuts, cuts[1:])]


def _popularity(c):
    n = c["adapters"]
    p = (np.arange(1, n + 1) ** -1.1) if c["zipf"] else np.ones(n)
    return p / p.sum()


def _tune_lengths(c):
    # the sequences of a case that tunes whole batches have one length; odd totals give ragged ones
    t, n = c["tune_rows"], c["tune_seqs"]
    return [t // n] * n if n and t % n == 0 else _lengths(t, n)


def _segments(c, seed):
    rng = np.random.default_rng(seed)
    n = c["adapters"]
    prompts = [(ln, int(a)) for ln, a in zip(_lengths(c["prompt_rows"], c["prompts"]), rng.integers(0, n, c["prompts"]))]
    dec = rng.choice(n, c["decode_rows"], p=_popularity(c))
    if c["by_adapter"]:
        dec = np.sort(dec)
    tune = [(ln, n - 1 - k % c["tune_adapters"]) for k, ln in enumerate(_tune_lengths(c))]
    decode_first = [(1, int(a)) for a in dec] + [(1, -1)] * c["base_rows"]
    segs, row = [], 0
    for flag, part in ((0, prompts), (0, decode_first), (1, tune)):
        for ln, a in part:
            segs.append((row, ln, a, flag))
            row += ln
    return synth.segments_array(segs), row


def _shapes(c):
    if c["kind"] == "projection":
        return {"p": (c["d_in"], c["d_out"])}
    d, f = c["hidden"], c["ffn"]
    kv = c["kv"] if c["kind"] == "set" else c["kv_heads"] * (d // c["heads"])
    return {"q": (d, d), "k": (d, kv), "v": (d, kv), "o": (d, d), "gate": (d, f), "up": (d, f), "down": (f, d)}


SHARED_INPUT = {"k": "q", "v": "q", "up": "gate"}


# ---- what a program holds before the call ---------------------------------------------------------
_session = None


def _context():
    global _session
    if _session is None:
        _session = Session(torch.cuda.current_device())
    return _session


class _Values:
    """Seeded normal values made on the GPU: X, dY ~ N(0, 1), W ~ N(0, d_in^-1/2), A, B ~ N(0, 0.02)."""

    def __init__(self, seed, dtype):
        self.g = torch.Generator(device="cuda").manual_seed(int(seed) & 0x7FFFFFFF)
        self.dtype = dtype

    def __call__(self, *shape, std=1.0):
        return (torch.randn(*shape, generator=self.g, device="cuda") * std).to(self.dtype)


def _adapter_ranks(c):
    if not c["own_ranks"]:
        return None
    return [min(OWN_RANKS[i % len(OWN_RANKS)], c["rank"]) for i in range(c["adapters"])]


def _adapters(c, v, d_in, d_out):
    n, r = c["adapters"], c["rank"]
    A, B = v(n, r, d_in, std=0.02), v(n, r, d_out, std=0.02)
    ranks = _adapter_ranks(c)
    if ranks:                                   # stored padded with zero rows
        keep = torch.arange(r, device="cuda")[None, :] < torch.tensor(ranks, device="cuda")[:, None]
        A *= keep[:, :, None]
        B *= keep[:, :, None]
    scale = torch.tensor([32.0 / x for x in (ranks or [16] * n)], dtype=torch.float32, device="cuda")
    return A, B, scale


class _Projection:
    """Weights, batch and buffers of one projection, and its calls."""

    def __init__(self, c, v, d_in, d_out, n_rows, plan, X=None):
        td, dev = torch_dtype(c["dtype"]), "cuda"
        self.W = v(d_in, d_out, std=d_in ** -0.5)
        self.A, self.B, self.scale = _adapters(c, v, d_in, d_out)
        self.layer = mb.make_layer(self.W, self.A, self.B, self.scale)
        self.X = v(n_rows, d_in) if X is None else X
        self.Y = torch.empty(n_rows, d_out, dtype=td, device=dev)
        self.x_save = self.u_save = self.dY = None
        t, r = c["tune_rows"], c["rank"]
        if t:
            n = len(mb.mlora_plan_ft_adapters(plan))
            self.x_save = torch.empty(t, d_in, dtype=td, device=dev)
            self.u_save = torch.empty(t, r, device=dev)
            self.dY = v(t, d_out)
            self.dX = torch.empty(t, d_in, dtype=td, device=dev)
            self.dA, self.dB = torch.empty(n, r, d_in, device=dev), torch.empty(n, r, d_out, device=dev)
        if c["update"]:
            slots = torch.tensor(mb.mlora_plan_ft_adapters(plan), device=dev)
            self.wA, self.wB = self.A[slots].float(), self.B[slots].float()
            self.mA, self.vA, self.mB, self.vB = (torch.zeros_like(t) for t in (self.wA, self.wA, self.wB, self.wB))
            self.step = 0

    def forward(self, ctx, plan):
        mb.mlora_mixed_forward(ctx, self.layer, plan, self.X, self.Y, self.x_save, self.u_save)

    def backward(self, ctx, plan):
        mb.mlora_backward(ctx, self.layer, plan, self.dY, self.x_save, self.u_save, self.dA, self.dB, self.dX)

    def update(self, ctx, plan):
        self.step += 1
        mb.mlora_adamw_update(ctx, self.layer, plan, self.dA, self.dB, self.wA, self.wB, self.mA, self.vA, self.mB, self.vB,
                              self.step)

    def outputs(self, c):
        out = [self.Y]
        if c["tune_rows"]:
            out += [self.x_save, self.u_save]
        if c["backward"]:
            out += [self.dA, self.dB, self.dX]
        if c["update"]:
            out += [self.wA, self.wB, self.mA, self.mB, self.vA, self.vB, self.A, self.B]
        return out


class _State:
    pass


def prepare(case, seed):
    c = dict(_DEFAULTS, **case)
    sess = _context()
    s = _State()
    s.case, s.ctx, s.seed = c, sess.ctx, int(seed)
    v = _Values(seed, torch_dtype(c["dtype"]))
    segs, rows = _segments(c, seed)
    if c["kind"] == "layer":
        p = {"g1": 1.0 + 0.1 * v(c["hidden"]).float(), "g2": 1.0 + 0.1 * v(c["hidden"]).float()}
        for name, (di, do) in _shapes(c).items():
            p["W_" + name] = v(di, do, std=di ** -0.5)
            p["A_" + name], p["B_" + name], p["s_" + name] = _adapters(c, v, di, do)
        s.layer = DecoderLayer(sess, p, c["heads"], c["kv_heads"], max_ft_rows=max(c["tune_rows"], 1))
        s.x, s.segs = v(rows, c["hidden"]), segs
        s.dy = v(c["tune_rows"], c["hidden"]) if c["backward"] else None
        return s
    ranks = _adapter_ranks(c)
    if ranks:
        s.plan = mb.mlora_plan_create_ranked(s.ctx, segs, rows, c["adapters"], ranks)
    else:
        s.plan = mb.mlora_plan_create(s.ctx, segs, rows, c["adapters"])
    weakref.finalize(s, mb.mlora_plan_destroy, s.plan)
    s.projections = {}
    for name, (di, do) in _shapes(c).items():
        other = s.projections.get(SHARED_INPUT.get(name))
        s.projections[name] = _Projection(c, v, di, do, rows, s.plan, None if other is None else other.X)
    return s


def run(s):
    c = s.case
    if c["kind"] == "layer":
        y = s.layer.forward(s.x, s.segs)
        if not c["backward"]:
            return [y]
        dx, grads, _slots = s.layer.backward(s.dy)
        return [y, dx, grads]
    if c["dropout"]:
        mb.mlora_set_dropout(s.ctx, c["dropout"], s.seed)
    for p in s.projections.values():
        p.forward(s.ctx, s.plan)
    if c["backward"]:
        for p in reversed(s.projections.values()):
            p.backward(s.ctx, s.plan)
            if c["update"]:
                p.update(s.ctx, s.plan)
    if c["dropout"]:
        mb.mlora_set_dropout(s.ctx, 0.0, 0)
    return [p.outputs(c) for p in s.projections.values()]


# ---- the same results in 64 bits ---------------------------------------------------------------------
class _Mixed64:
    """`X W + s (X A^T) B` per row of one batch, its gradients and the update, in torch float64."""

    def __init__(self, c, seed):
        segs, self.rows = _segments(c, seed)
        self.first = self.rows - c["tune_rows"]                     # fine-tuning rows are the last ones, in save order
        row_adapter = np.full(self.rows, -1)
        for start, n, a, _ in segs:
            row_adapter[start:start + n] = a
        self.sequences = [(int(s), int(n)) for s, n, _, _ in segs if n > 0]
        self.row_adapter = row_adapter
        self.slots = list(dict.fromkeys(int(a) for _, n, a, flag in segs if flag and n > 0))
        self.keep = None
        if c["dropout"]:
            self.keep = _kept(int(seed), c["tune_rows"], c["d_in"], c["dropout"]) / (1.0 - c["dropout"])

    def groups(self, first=0, slots=None):
        ids = self.row_adapter[first:]
        for a in (sorted(set(ids[ids >= 0].tolist())) if slots is None else slots):
            yield a, torch.from_numpy(np.flatnonzero(ids == a)).cuda()

    def linear(self, x, W, A, B, scale, first=0):
        """`x` holds the rows from `first` on; differentiable in x, A and B."""
        y = x @ W
        for a, at in self.groups(first):
            y = y.index_add(0, at, scale[a] * ((x[at] @ A[a].T) @ B[a]))
        return y

    def projection(self, c, p):
        W, A, B, scale, X = (t.double() for t in (p.W, p.A, p.B, p.scale, p.X))
        f = self.first
        branch = X.clone()
        if self.keep is not None:
            branch[f:] *= self.keep
        U = X.new_zeros(self.rows, c["rank"])
        Y = X @ W
        for a, at in self.groups():
            U[at] = branch[at] @ A[a].T
            Y[at] += scale[a] * (U[at] @ B[a])
        out = [Y]
        if c["tune_rows"]:
            out += [X[f:], U[f:]]
        if c["backward"]:
            dY = p.dY.double()
            dX = dY @ W.T
            dA, dB = [], []
            for a, at in self.groups(f, self.slots):
                V = scale[a] * (dY[at] @ B[a].T)
                low = V @ A[a]
                dX[at] += low if self.keep is None else low * self.keep[at]
                dA.append(V.T @ branch[f:][at])
                dB.append(scale[a] * (U[f:][at].T @ dY[at]))
            out += [torch.stack(dA), torch.stack(dB), dX]
        if c["update"]:
            lr, b1, b2, eps, wd = 1e-3, 0.9, 0.999, 1e-8, 0.01      # the defaults of mlora_adamw_update
            new, moments = [], []
            for all_rows, grads in ((A, out[3]), (B, out[4])):
                w = all_rows[self.slots]
                m, v = (1 - b1) * grads, (1 - b2) * grads * grads
                w = w - lr * wd * w - lr * (m / (1 - b1)) / ((v / (1 - b2)).sqrt() + eps)
                all_rows[self.slots] = w
                new.append(w)
                moments.append((m, v))
            (mA, vA), (mB, vB) = moments
            out += [*new, mA, mB, vA, vB, A, B]
        return out


def _kept(seed, rows, d_in, p):
    """The dropout mask of mlora.h: field k & 3 of output (m << 32 | k >> 2) + 1 of a SplitMix64 stream, for element (m, k)."""
    u = np.uint64
    with np.errstate(over="ignore"):
        z = (np.arange(rows, dtype=u)[:, None] << u(32)) | np.arange((d_in + 3) // 4, dtype=u)[None, :]
        z = u(seed) + (z + u(1)) * u(0x9E3779B97F4A7C15)
        z = (z ^ (z >> u(30))) * u(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> u(27))) * u(0x94D049BB133111EB)
        z = z ^ (z >> u(31))
    fields = np.stack([(z >> u(16 * j)) & u(0xFFFF) for j in range(4)], axis=-1).reshape(rows, -1)[:, :d_in]
    return torch.from_numpy((fields >= u(round(p * 65536))).astype(np.float64)).cuda()


def _layer64(b, x, w, n_heads, n_kv, first=0):
    """A decoder layer over the rows from `first` on: norm eps 1e-5, rotary base 500000 on halves, causal attention in a sequence."""
    T, d = x.shape
    dh = d // n_heads

    def norm(t, g):
        return t * torch.rsqrt((t * t).mean(-1, keepdim=True) + 1e-5) * g

    def lin(name, t):
        return b.linear(t, *(w[k + name].double() if k in ("W_", "s_") else w[k + name] for k in ("W_", "A_", "B_", "s_")), first)

    seqs = [(s - first, n) for s, n in b.sequences if s >= first]
    pos = torch.cat([torch.arange(n) for _, n in seqs]).double().cuda()
    inv = 500000.0 ** (-torch.arange(dh // 2, device="cuda", dtype=torch.float64) * 2.0 / dh)
    cos, sin = torch.cos(pos[:, None] * inv)[:, None], torch.sin(pos[:, None] * inv)[:, None]

    def rope(t):
        lo, hi = t[..., :dh // 2], t[..., dh // 2:]
        return torch.cat([lo * cos - hi * sin, hi * cos + lo * sin], -1)

    h1 = norm(x, w["g1"])
    q, k, v = (lin(n, h1).view(T, -1, dh) for n in "qkv")
    q, k = rope(q), rope(k)
    parts = []
    for s, n in seqs:                                              # in row order: every row is in one sequence
        qs, ks, vs = (t[s:s + n].transpose(0, 1) for t in (q, k, v))
        ks, vs = (t.repeat_interleave(n_heads // n_kv, 0) for t in (ks, vs))
        score = (qs @ ks.transpose(1, 2) / math.sqrt(dh)).masked_fill(torch.ones(n, n, device="cuda").triu(1).bool(), -math.inf)
        parts.append((score.softmax(-1) @ vs).transpose(0, 1).reshape(n, d))
    x2 = x + lin("o", torch.cat(parts))
    h2 = norm(x2, w["g2"])
    return x2 + lin("down", torch.nn.functional.silu(lin("gate", h2)) * lin("up", h2))


def exact(case, seed):
    """What `run` returns on a state just prepared, from the definitions in 64 bits."""
    c = dict(_DEFAULTS, **case)
    s = prepare(case, seed)
    b = _Mixed64(c, seed)
    if c["kind"] != "layer":
        return [b.projection(c, p) for p in s.projections.values()]
    layer, w = s.layer, {"g1": s.layer.g1.double(), "g2": s.layer.g2.double()}
    for name, p in layer.proj.items():
        w["W_" + name], w["A_" + name], w["B_" + name], w["s_" + name] = p.W, p.A.double(), p.B.double(), p.scale
    x = s.x.double()
    with torch.no_grad():
        y = _layer64(b, x, w, c["heads"], c["kv_heads"])
    if not c["backward"]:
        return [y]
    f = b.first
    leaf = x[f:].clone().requires_grad_(True)
    wanted = [w[k + n].requires_grad_(True) for n in layer.proj for k in ("A_", "B_")]
    with torch.enable_grad():
        got = torch.autograd.grad(_layer64(b, leaf, w, c["heads"], c["kv_heads"], f), [leaf] + wanted, s.dy.double())
    grads = {n: (got[1 + 2 * i][b.slots], got[2 + 2 * i][b.slots]) for i, n in enumerate(layer.proj)}
    return [y, got[0], grads]


# ---- the work of a case and how exact its results are ----------------------------------------------
def _distinct(c):
    """Adapters that a batch meets, in the mean over seeds."""
    p = _popularity(c)
    missed = (1 - p) ** c["decode_rows"] * (1 - 1 / len(p)) ** c["prompts"]
    tuned = np.zeros(len(p), dtype=bool)
    for k in range(len(_tune_lengths(c))):
        tuned[len(p) - 1 - k % c["tune_adapters"]] = True
    return float(np.where(tuned, 1.0, 1 - missed).sum()), int(tuned.sum())


def work(case):
    c = dict(_DEFAULTS, **case)
    e = 2 if c["dtype"] == "bf16" else 4
    t = c["tune_rows"]
    rows = c["prompt_rows"] + c["decode_rows"] + c["base_rows"] + t
    lora_rows = rows - c["base_rows"]
    used, slots = _distinct(c)
    ranks = _adapter_ranks(c)
    r = float(np.mean(ranks)) if ranks else c["rank"]
    layer = c["kind"] == "layer"
    nbytes = flops = 0.0
    for name, (di, do) in _shapes(c).items():
        base, low = 2.0 * di * do, 2.0 * r * (di + do)
        flops += rows * base + lora_rows * low
        nbytes += e * (di * do + used * r * (di + do))
        if c["backward"]:
            flops += t * base + 2 * t * low                     # dX; V and its expand, dA and dB
            nbytes += 4 * slots * c["rank"] * (di + do)
            if layer:                                           # the recompute, without the last product's base part
                flops += t * (base if name != "down" else 0) + t * (low if name != "down" else 2.0 * r * di)
        if c["update"]:
            nbytes += 4 * 6 * slots * c["rank"] * (di + do) + e * slots * c["rank"] * (di + do)
        if not layer:
            nbytes += e * rows * (do + (0 if name in SHARED_INPUT else di))
            if t:
                nbytes += e * t * di + 4 * t * c["rank"]        # x_save, u_save
            if c["backward"]:
                nbytes += e * t * (di + do)                     # dY, dX
    if layer:
        pairs = sum(n * (n + 1) / 2 for n in _lengths(c["prompt_rows"], c["prompts"])) + c["decode_rows"] + c["base_rows"]
        tuned = sum(n * (n + 1) / 2 for n in _tune_lengths(c))
        attn = 4.0 * c["hidden"]
        flops += attn * (pairs + tuned)
        nbytes += e * 2 * rows * c["hidden"]
        if c["backward"]:
            flops += 3.5 * attn * tuned                         # recompute, then five products against two
            nbytes += e * 2 * t * c["hidden"]
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    # Measured between the library's own kernel variants (other orders of sums, other operand roundings) on the same inputs:
    # projections differ by up to 2.4e-4 and by one bf16 step (0.0078) at the most; storing a product in bf16 alone moves it
    # 1.7e-3 from its 64-bit value, which is what the two roundings of an input gradient under dropout can show.  A layer is a
    # dozen such roundings in series: up to 3.9e-3 and 0.038.
    if case.get("dtype") == "f32":
        return {"rel": 1e-5}
    if case.get("kind") == "layer":
        return {"rel": 1.6e-2, "max": 0.15}
    return {"rel": 4e-3, "max": 0.03}
