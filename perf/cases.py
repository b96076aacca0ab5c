"""The work a streaming video DiT has this library do, as measurable cases.

A program that denoises video chunk by chunk keeps, for each transformer
layer, a cache of rotated keys and values per (chunk, level) state with its
split workspace, and a node table per pipeline round.  Its calls per layer and
round are:

  layer        x -> q, k, v (projection), RoPE + cache write, attention: either
               with the RoPE and the write fused into the projection, or, in
               models that normalise q and k, as projection, fused
               RMSNorm + RoPE + write, and attention;
  attend       attention alone (a program whose own code makes q, k, v),
               dense, frame-causal, block-sparse or with token masks;
  write        the RoPE + cache write alone (the clean-state refresh and the
               prefill of history: keys and values, no queries), with or
               without the normalisation;
  project      the projection alone, or fused with RoPE and the write.

The sizes are those of the repository's workloads (Wan2.1-like chunks of 3
latent frames of 30 x 52 patches, 12 or 40 heads of 128; tiny test chunks) and
generic ones between them: low-resolution and single-frame chunks, 64-wide
heads, tokens that do not divide by the tile sizes.
"""
from __future__ import annotations

import math

import torch

from paper_2609_22283_gb300 import sva

LEVELS = 4       # denoising levels of the pipelines (level 0 = clean)
EPS = 1e-6       # of the q/k normalisation
DEV = "cuda"


def _case(name=None, **kw):
    """A case with every field set.

    kind     "layer", "layer_norm", "attend", "write", "write_norm", "project", "project_rope"
    F,Hp,Wp  latent frames of a chunk, patch rows and columns of a frame
    H,d      heads and head dimension;  C: input features of the projection
    streams  independent videos, `nodes` nodes (consecutive levels of one pipeline round) in each
    W        history chunks a node reads;  policy "clean", "same" or "prog"
    causal   frame-causal attention inside the own chunk
    mask     "", "tiles" (block-sparse: each block of `span` query tiles keeps its own chunk and
             a share `keep` of the history's key tiles), "local" (token masks: a query sees the
             keys, of its own chunk and of the history, within `span` patch rows and columns),
             "random" (token masks: a query keeps each key with probability one half)
    """
    c = dict(kind="attend", F=3, Hp=30, Wp=52, H=12, d=128, C=0, streams=1, nodes=1, W=3, policy="prog",
             causal=False, mask="", span=0, keep=1.0)
    c.update(kw)
    if not c["C"]:
        c["C"] = c["H"] * c["d"]
    if name is not None:
        c["name"] = name
    return c


def listed():
    return [
        # The smallest call: the repository's tiny workload (2 nodes of 64 tokens, 2 heads of 64) as one
        # layer; what counts is launches and latency, as in tests, previews and a distilled model's layers.
        _case("layer tiny", kind="layer", F=1, Hp=8, Wp=8, H=2, d=64, nodes=2, W=2),
        # A single-frame low-resolution chunk (320 tokens, the last tile half full) through a whole layer of
        # a 12-head model that normalises q and k: an interactive session's call, too small to fill the GPU.
        _case("layer small", kind="layer_norm", F=1, Hp=16, Wp=20, policy="clean"),
        # One denoising update of the serial, clean-history schedule: a whole layer of the 12-head model on
        # one full-size chunk (4680 tokens) with normalised q and k.
        _case("layer serial", kind="layer_norm", policy="clean"),
        # The pipelined schedule's round: 4 nodes of 4680 tokens, 6 history chunks each.
        _case("attend round", nodes=4, W=6),
        # The largest call: two videos' rounds batched, 8 nodes of a 40-head model.
        _case("attend large", H=40, streams=2, nodes=4, W=6),
        # 64-wide heads (smaller DiTs), mid-size chunks of 2160 tokens, two nodes, same-level history.
        _case("attend narrow", Hp=20, Wp=36, H=16, d=64, nodes=2, W=4, policy="same"),
        # The first chunk of a video: no history yet, frame-causal inside the chunk.
        _case("attend first", W=0, causal=True),
        # Query-dependent block-sparse history: each 256-query block keeps half of the history's tiles.
        _case("attend sparse", nodes=4, W=6, mask="tiles", span=2, keep=0.5),
        # Spatially local attention by token masks (own chunk and history), one full-size chunk.
        _case("attend local", W=3, mask="local", span=6),
        # The clean-state refresh of a 40-head model: one chunk's keys (normalised) and values into the cache.
        _case("write clean", kind="write_norm", H=40),
        # A round's states written without normalisation: bandwidth alone.
        _case("write round", kind="write", nodes=4),
        # The projection of one full-size chunk of the 40-head model, RoPE and cache write fused in.
        _case("project large", kind="project_rope", H=40),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["layer", "layer_norm", "attend", "attend", "attend", "write", "write_norm", "project",
                       "project_rope"])
    d = rng.choice([64, 128, 128])
    H = _log(rng, 2, 40)
    if d == 64 and H % 2:
        H += 1       # the projection's outputs come in multiples of 128
    c = _case(kind=kind, F=rng.randint(1, 4), Hp=_log(rng, 5, 32), Wp=_log(rng, 5, 52), H=H, d=d,
              streams=rng.choice([1, 1, 1, 2]), nodes=rng.randint(1, 4), W=rng.randint(0, 6),
              policy=rng.choice(["clean", "same", "prog"]))
    if kind.startswith(("layer", "project")) and rng.random() < 0.3:
        c["C"] = 8 * _log(rng, 16, 640)
    if kind == "attend":
        c["causal"] = rng.random() < 0.25
        c["mask"] = rng.choice(["", "", "", "tiles", "local", "random"])
        if c["mask"] == "tiles":
            c["span"], c["keep"] = rng.choice([1, 2, 2, 4]), round(rng.uniform(0.1, 0.9), 2)
        if c["mask"] == "local":
            c["span"] = rng.randint(2, 10)
        if c["mask"] in ("local", "random"):
            c["streams"] = 1
    return c


# ------------------------------------------------------------------ the round

def _tokens(c):
    return c["F"] * c["Hp"] * c["Wp"]


def _pairs(d):
    hw = d // 6
    return (d // 2 - 2 * hw, hw, hw)


def _round(c):
    """[(node, its history states)] in order, states as (seq, chunk, level)."""
    last = c["W"] + c["nodes"]
    phi = {"clean": lambda j, r: 0, "same": lambda j, r: j, "prog": lambda j, r: max(j - r, 0)}[c["policy"]]
    out = []
    for s in range(c["streams"]):
        for i in range(c["nodes"]):
            b, j = last - i, LEVELS - i
            out.append(((s, b, j), [(s, b - r, phi(j, r)) for r in range(1, min(c["W"], b - 1) + 1)]))
    return out


def _states(c):
    """(the nodes' own states, the other states they read)."""
    own = [n for n, _ in _round(c)]
    seen, other = set(own), []
    for _, ctx in _round(c):
        for s in ctx:
            if s not in seen:
                seen.add(s)
                other.append(s)
    return own, other


def _local_1d(n, span):
    i = torch.arange(n)
    return (i[:, None] - i[None, :]).abs() <= span


def _local(c):
    """bool [T][T]: patches within `span` rows and columns, whatever their frame."""
    h, w = _local_1d(c["Hp"], c["span"]).to(DEV), _local_1d(c["Wp"], c["span"]).to(DEV)
    hw = (h[:, None, :, None] & w[None, :, None, :]).reshape(c["Hp"] * c["Wp"], -1)
    return hw.repeat(c["F"], c["F"])


def _pack(keep):
    """bool [..., n] -> int32 [..., ceil(n / 32)], bit k % 32 of word k // 32."""
    n = keep.shape[-1]
    words = -(-n // 32)
    k = torch.zeros(keep.shape[:-1] + (words * 32,), dtype=torch.bool, device=keep.device)
    k[..., :n] = keep
    v = k.view(keep.shape[:-1] + (words, 32)).long() << torch.arange(32, device=keep.device)
    v = v.sum(-1)
    return torch.where(v >= 2 ** 31, v - 2 ** 32, v).to(torch.int32)


def _unpack(words, n):
    b = (words.unsqueeze(-1) >> torch.arange(32, device=words.device, dtype=torch.int32)) & 1
    return b.reshape(words.shape[:-1] + (-1,))[..., :n].bool()


class _Inputs:
    """What the calls take, from the seed alone: tensors on the GPU, masks included."""

    def __init__(self, c, seed):
        g = torch.Generator(device=DEV)
        g.manual_seed(int(seed))
        T, H, d = _tokens(c), c["H"], c["d"]
        self.own, self.other = _states(c)
        n, kind = len(self.own), c["kind"]

        def normal(*shape, by=1.0, dtype=torch.bfloat16):
            return (torch.randn(shape, generator=g, device=DEV) * by).to(dtype)

        if kind.startswith(("layer", "project")):
            self.x = normal(n, T, c["C"])
            self.w = normal(3 * H * d, c["C"], by=c["C"] ** -0.5)
            self.b = normal(3 * H * d, by=0.1, dtype=torch.float32)
        if kind.endswith("norm"):
            self.gk = torch.rand(H * d, generator=g, device=DEV) + 0.5
            self.gq = torch.rand(H * d, generator=g, device=DEV) + 0.5
        if kind.startswith("write"):
            self.k, self.v = normal(n, T, H, d), normal(n, T, H, d)
        self.kv = {}
        if kind.startswith(("layer", "attend")):
            for s in self.other + (self.own if kind == "attend" else []):
                self.kv[s] = (normal(T, H, d), normal(T, H, d))
        if kind == "attend":
            self.q = normal(n, T, H, d)
        # masks
        self.tile = self.tok_own = self.tok_hist = None
        W, words = max(c["W"], 1), -(-T // 32)
        if c["mask"] == "tiles":
            nt = -(-T // 128)
            rows = -(-nt // c["span"])
            keep = torch.rand((n, rows, (1 + c["W"]) * nt), generator=g, device=DEV) < c["keep"]
            keep = keep.repeat_interleave(c["span"], dim=1)[:, :nt]
            keep[:, :, :nt] = True
            self.tile = _pack(keep)
        elif c["mask"] == "local":
            m = _pack(_local(c))
            self.tok_own = m.expand(n, T, words).contiguous()
            self.tok_hist = m[None, :, None, :].expand(n, T, W, words).contiguous()
        elif c["mask"] == "random":
            def bits(*shape):
                return torch.randint(-2 ** 31, 2 ** 31, shape, generator=g, device=DEV, dtype=torch.int64).to(torch.int32)
            self.tok_own, self.tok_hist = bits(n, T, words), bits(n, T, W, words)
            u = torch.arange(T, device=DEV)   # a query sees itself
            bit = torch.ones_like(u) << (u % 32)
            bit = torch.where(bit >= 2 ** 31, bit - 2 ** 32, bit).to(torch.int32)
            self.tok_own[:, u, u // 32] |= bit


class _State:
    pass


def _geometry(c, own, other):
    top = max(b for _, b, _ in own + other)
    return sva.make_geometry(c["H"], c["d"], c["F"], c["Hp"], c["Wp"], num_slots=len(own) + len(other),
                             pairs=_pairs(c["d"]), max_frames=c["F"] * (top + 2))


def prepare(case, seed):
    """A layer's cache with its workspace and filled history, the round's node table, the inputs and
    the output buffers a program reuses from round to round."""
    c, s = case, _State()
    s.c, s.i = c, _Inputs(c, seed)
    i = s.i
    own, other = i.own, i.other
    T, H, d, n = _tokens(c), c["H"], c["d"], len(own)
    s.cache = sva.Cache(_geometry(c, own, other), device=torch.device(DEV))
    s.cache.set_workspace(torch.empty(s.cache.workspace_bytes(), dtype=torch.uint8, device=DEV))
    slot = {st: s.cache.bind(*st) for st in own + other}
    within = sva.WITHIN_FRAME_CAUSAL if c["causal"] else sva.WITHIN_BIDIRECTIONAL
    s.nodes = sva.make_nodes([dict(seq=q, chunk=b, level=j, own_slot=slot[(q, b, j)],
                                   ctx=[slot[t] for t in ctx], within=within)
                              for (q, b, j), ctx in _round(c)])
    for st in list(i.kv):    # history (and, for attention alone, the nodes' own states)
        k, v = i.kv[st]
        s.cache.rope_kv_write([dict(seq=st[0], chunk=st[1], level=st[2], own_slot=slot[st])], k[None], v[None])
        del i.kv[st]
    if not c["kind"].startswith("write"):
        s.q = i.q if c["kind"] == "attend" else torch.empty((n, T, H, d), dtype=torch.bfloat16, device=DEV)
    if c["kind"] in ("layer_norm", "project"):
        s.k, s.v = torch.empty_like(s.q), torch.empty_like(s.q)
    if c["kind"].startswith(("layer", "attend")):
        s.out = torch.empty_like(s.q)
        s.lse = torch.empty((n, H, T), dtype=torch.float32, device=DEV)
    pool = s.cache.slot_pool()
    s.written = [pool[slot[st]][:, :, :T] for st in own]   # K' and V of the nodes' own states, in the cache
    return s


def run(state):
    s, i, c = state, state.i, state.c
    kind = c["kind"]
    if kind == "write":
        s.cache.rope_kv_write(s.nodes, i.k, i.v)
        return s.written
    if kind == "write_norm":
        s.cache.rope_kv_write_qknorm(s.nodes, i.k, i.v, None, i.gk, None, EPS)
        return s.written
    if kind == "project":
        s.cache.qkv_project(i.x, i.w, i.b, s.q, s.k, s.v)
        return [s.q, s.k, s.v]
    if kind == "project_rope":
        s.cache.qkv_project_rope(s.nodes, i.x, i.w, i.b, s.q)
        return [s.q] + s.written
    if kind == "layer":
        s.cache.qkv_project_rope(s.nodes, i.x, i.w, i.b, s.q)
    elif kind == "layer_norm":
        s.cache.qkv_project(i.x, i.w, i.b, s.q, s.k, s.v)
        s.cache.rope_kv_write_qknorm(s.nodes, s.k, s.v, s.q, i.gk, i.gq, EPS)
    if c["mask"] == "":
        s.cache.attend_nodes(s.nodes, s.q, s.out, s.lse)
    elif c["mask"] == "tiles":
        s.cache.attend_nodes_sparse(s.nodes, s.q, s.out, i.tile, s.lse)
    else:
        s.cache.attend_nodes_masked(s.nodes, s.q, s.out, s.lse, own_mask=i.tok_own,
                                    hist_mask=i.tok_hist if c["W"] else None)
    return [s.out, s.lse]


# ------------------------------------------------------------------ work and tolerance

def _visible(c):
    """(query, key) pairs that may attend, over all nodes and one head."""
    T, F, hw = _tokens(c), c["F"], c["Hp"] * c["Wp"]
    near = 1.0
    if c["mask"] == "random":
        near = 0.5
    elif c["mask"] == "local":
        near = float(_local_1d(c["Hp"], c["span"]).double().mean() * _local_1d(c["Wp"], c["span"]).double().mean())
    keep = c["keep"] if c["mask"] == "tiles" else 1.0
    own = (hw * hw * F * (F + 1) / 2 if c["causal"] else T * T) * near
    return sum(own + len(ctx) * T * T * near * keep for _, ctx in _round(c))


def work(case):
    c, kind = case, case["kind"]
    T, N = _tokens(c), c["H"] * c["d"]
    own, other = _states(c)
    rows = len(own) * T
    by, fl = 0.0, 0.0
    if kind.startswith(("layer", "project")):
        by += 2 * rows * c["C"] + 2 * 3 * N * c["C"] + 4 * 3 * N
        fl += 2 * rows * c["C"] * 3 * N
    if kind in ("project", "project_rope"):
        by += 2 * 3 * rows * N
    if kind.startswith("layer"):
        by += 2 * 2 * rows * N       # the new states' K and V into the cache
    if kind.startswith("write"):
        by += 2 * 4 * rows * N
    if kind.endswith("norm"):
        by += 4 * N * (1 if kind == "write_norm" else 2)
    if kind.startswith(("layer", "attend")):
        held = len(other) + (len(own) if kind == "attend" else 0)
        by += 2 * 2 * held * T * N + 2 * rows * N + 4 * rows * c["H"]
        if kind == "attend":
            by += 2 * rows * N       # the queries
        if c["mask"] in ("local", "random"):
            by += rows * T / 8 + sum(T * T * len(ctx) / 8 for _, ctx in _round(c))
        fl += 4.0 * _visible(c) * N
    return {"bytes": by, "flops": fl}


def tolerance(case):
    kind = case["kind"]
    if kind.startswith("write"):
        return {"rel": 2e-3, "max": 2e-2}     # one bf16 rounding of a 32-bit rotation
    if kind.startswith("project"):
        return {"rel": 7e-3, "max": 4e-2}     # 32-bit sums, one bf16 rounding
    return {"rel": 1.5e-2, "max": 0.15}       # bf16 weights of the values, bf16 results


# ------------------------------------------------------------------ in 64 bits

def _rope(c, x, chunk):
    """x [T][H][d] rotated at the chunk's positions, in 64 bits."""
    T, d = _tokens(c), c["d"]
    u = torch.arange(T, device=DEV)
    hw = c["Hp"] * c["Wp"]
    at = (c["F"] * chunk + u // hw, u % hw // c["Wp"], u % c["Wp"])
    angles = []
    for pos, p in zip(at, _pairs(d)):
        f = 10000.0 ** (-torch.arange(p, device=DEV, dtype=torch.float64) / p)
        angles.append(pos.double()[:, None] * f)
    a = torch.cat(angles, dim=1)[:, None, :]
    y = x.double().reshape(T, -1, d // 2, 2)
    co, si = torch.cos(a), torch.sin(a)
    return torch.stack((y[..., 0] * co - y[..., 1] * si, y[..., 0] * si + y[..., 1] * co), dim=-1).reshape(T, -1, d)


def _norm(x, gamma):
    """RMS normalisation of [T][H][d] over H * d, in 64 bits."""
    y = x.double().reshape(x.shape[0], -1)
    return (y * torch.rsqrt((y * y).mean(1, keepdim=True) + EPS) * gamma.double()).reshape(x.shape)


def exact(case, seed):
    c, kind = case, case["kind"]
    T, H, d, N = _tokens(c), c["H"], c["d"], c["H"] * c["d"]
    if work(c)["flops"] > 4.5e12:
        return None      # tens of seconds of 64-bit products
    i = _Inputs(c, seed)
    rnd = _round(c)
    if kind.startswith("write"):
        got = []
        for n, (_, b, _) in enumerate(i.own):
            k = _norm(i.k[n], i.gk) if kind == "write_norm" else i.k[n]
            got.append(torch.stack((_rope(c, k, b).transpose(0, 1), i.v[n].double().transpose(0, 1))))
        return got
    new_k, new_v, q = {}, {}, []
    if kind.startswith(("layer", "project")):
        wd, qs, ks, vs = i.w.double().t(), [], [], []
        for n, st in enumerate(i.own):
            y = (i.x[n].double() @ wd + i.b.double()).reshape(T, 3, H, d)
            a, k, v = y[:, 0], y[:, 1], y[:, 2]
            if kind == "layer_norm":
                a, k = _norm(a, i.gq), _norm(k, i.gk)
            if kind != "project":
                a, k = _rope(c, a, st[1]), _rope(c, k, st[1])
            qs.append(a), ks.append(k), vs.append(v)
            new_k[st], new_v[st] = k, v
        if kind == "project":
            return [torch.stack(qs), torch.stack(ks), torch.stack(vs)]
        if kind == "project_rope":
            return [torch.stack(qs)] + [torch.stack((k.transpose(0, 1), v.transpose(0, 1))) for k, v in zip(ks, vs)]
        q = qs
    else:
        q = [i.q[n].double() for n in range(len(i.own))]
    for st, (k, v) in i.kv.items():      # states held in bf16, rotated and rounded once
        new_k[st], new_v[st] = _rope(c, k, st[1]).bfloat16(), v
    out = torch.empty((len(rnd), T, H, d), dtype=torch.float64, device=DEV)
    lse = torch.empty((len(rnd), H, T), dtype=torch.float64, device=DEV)
    for n, (st, ctx) in enumerate(rnd):
        see = [st] + ctx
        hide = None
        if c["causal"] or c["mask"]:
            keep = torch.ones((T, len(see) * T), dtype=torch.bool, device=DEV)
            if c["causal"]:
                f = torch.arange(T, device=DEV) // (c["Hp"] * c["Wp"])
                keep[:, :T] &= f[:, None] >= f[None, :]
            if c["mask"] == "tiles":
                nt = -(-T // 128)
                t = _unpack(i.tile[n], (1 + c["W"]) * nt).repeat_interleave(128, 0)[:T]
                for j in range(len(see)):
                    keep[:, j * T:(j + 1) * T] &= t[:, j * nt:(j + 1) * nt].repeat_interleave(128, 1)[:, :T]
            elif c["mask"]:
                keep[:, :T] &= _unpack(i.tok_own[n], T)
                for j in range(len(ctx)):
                    keep[:, (j + 1) * T:(j + 2) * T] &= _unpack(i.tok_hist[n, :, j], T)
            hide = ~keep
        for h in range(H):
            k = torch.cat([new_k[t][:, h].double() for t in see])
            v = torch.cat([new_v[t][:, h].double() for t in see])
            for r in range(0, T, 2048):
                s = (q[n][r:r + 2048, h] @ k.t()) / math.sqrt(d)
                if hide is not None:
                    s.masked_fill_(hide[r:r + 2048], -math.inf)
                l = torch.logsumexp(s, dim=1)
                s.sub_(torch.where(l == -math.inf, 0.0, l)[:, None]).exp_()
                out[n, r:r + 2048, h] = s @ v
                lse[n, h, r:r + 2048] = l
    return [out, lse]
