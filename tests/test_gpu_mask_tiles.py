"""Token masks and the running max: keys far larger than the rest (their
logits are hundreds of log2 units above the others') that a mask hides from
some queries only.  A tile whose unmasked maximum jumps past the rescale
threshold must take the maximum over what the row sees, and one that does not
must leave the running max alone; rows that see nothing, whole tiles that are
visible, hidden or partly hidden, and ragged last tiles, at both head
dimensions.

Reference: the same op in fp64 torch on the rotated Q and the K', V the cache
holds, with the bound of the rounding of P and of the output, and of fp32
logits below 2^12 log2 units (an error of 2^-10, which scales the weights):
|d| <= 2^-8 (E_p|V| + |O|) + 2^-9 E_p|V|, and 2^-20 for the fp32 sums."""
import math

import pytest
import torch

from paper_2609_22283_gb300 import sva
from paper_2609_22283_gb300.inputs import pack_bits, rope_pairs_for

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("split", [False, True])
@pytest.mark.parametrize("T,W,pattern", [(130, 1, "random"), (256, 2, "blocks"), (300, 2, "random"),
                                         (520, 1, "blocks"), (97, 0, "random")])
def test_hidden_large_keys(T, W, pattern, d, split):
    H = 2
    cache = sva.Cache(sva.make_geometry(H, d, 1, 1, T, num_slots=W + 1, pairs=rope_pairs_for(d),
                                        max_frames=W + 4))
    if split:
        cache.set_workspace(torch.empty(cache.workspace_bytes(), dtype=torch.uint8, device="cuda"))
    gen = torch.Generator().manual_seed(T * 7 + W)
    slots = []
    large = (torch.arange(T) % 7 == 3) | (torch.arange(T) // 64 % 3 == 2)   # large keys of every state
    for b in range(W, -1, -1):
        k = torch.randn((1, T, H, d), generator=gen)
        k[0, large] *= 40.0 * (W + 1 - b)
        s = cache.bind(0, b + 1, 0)
        cache.rope_kv_write([dict(seq=0, chunk=b + 1, level=0, own_slot=s)], k.bfloat16().cuda(),
                            torch.randn((1, T, H, d), generator=gen).bfloat16().cuda())
        slots.append(s)
    nodes = sva.make_nodes([dict(seq=0, chunk=W + 1, level=0, own_slot=slots[0], ctx=slots[1:])])
    q = torch.randn((1, T, H, d), generator=gen).bfloat16().cuda()

    def mask():
        if pattern == "blocks":   # blocks of 96 x 160: whole tiles visible, hidden or cut
            m = torch.rand((T // 96 + 1, T // 160 + 1), generator=gen) < 0.6
            return m.repeat_interleave(96, 0)[:T].repeat_interleave(160, 1)[:, :T]
        m = torch.rand((T, T), generator=gen) < 0.5
        m[torch.arange(T) % 2 == 0] &= ~large      # every other query sees no large key
        m[5] = False                               # a query that sees nothing
        return m

    own, hist = mask(), torch.stack([mask() for _ in range(max(W, 1))], dim=1)   # [T][W][T]
    words = -(-T // 32)
    out, lse = torch.empty_like(q), torch.empty((1, H, T), dtype=torch.float32, device="cuda")
    cache.attend_nodes_masked(nodes, q, out, lse, own_mask=pack_bits(own[None], words).cuda(),
                              hist_mask=pack_bits(hist[None], words).cuda() if W else None)
    assert cache.poll() == sva.OK
    pool = cache.slot_pool()
    k = torch.cat([pool[s, 0, :, :T] for s in slots], dim=1).double()
    v = torch.cat([pool[s, 1, :, :T] for s in slots], dim=1).double()
    see = torch.cat([own] + [hist[:, j] for j in range(W)], dim=1).cuda()
    s = torch.einsum("thd,hkd->htk", q[0].double(), k) / math.sqrt(d)
    s.masked_fill_(~see, -math.inf)
    p = torch.nan_to_num(torch.softmax(s, dim=-1), nan=0.0)
    o, ev = torch.einsum("htk,hkd->thd", p, v), torch.einsum("htk,hkd->thd", p, v.abs())
    bound = 2.0 ** -8 * (ev + o.abs()) + 2.0 ** -9 * ev + 2.0 ** -20
    bad = ~((out[0].double() - o).abs() <= bound)
    assert not bad.any(), f"{int(bad.sum())} of {bad.numel()} elements out of bound"
    ref = torch.logsumexp(s, dim=-1)
    none = ref == -math.inf
    assert (lse[0][none] == -math.inf).all()
    assert ((lse[0].double() - ref)[~none].abs() <= 2e-3 + 2.0 ** -20 * ref[~none].abs()).all()
    cache.close()


# Launches long enough for the masks to be scanned for empty key tiles first (with a workspace)
# against the same call without a workspace, which walks every tile: T = 2500 (20 tiles, the last of
# 68 rows; 78.1 mask words), 12 heads, one or two nodes.  Both paths multiply the same tiles that
# hold a visible key, so they differ by the key-range split alone: two bf16 roundings of O and the
# rounding of P relative to another maximum.
SCAN_FORMS = {
    "both": {},
    "own only": {"hist": False},
    "history only": {"own": False},
    "hidden context": {"visible": [1, 0, 1, 1]},
    "long rows": {"extra": 3, "states": 6},
    "tile mask too": {"tiles": True},
    "frame causal": {"causal": True},
    "two nodes": {"n": 2},
}


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("form", sorted(SCAN_FORMS))
def test_scan_of_empty_tiles(form, d):
    f = SCAN_FORMS[form]
    F, Hp, Wp, H, W, n = 4, 25, 25, 12, 4, f.get("n", 1)
    T, nt = F * Hp * Wp, 20
    assert H * n * 10 * (W + 1) * nt >= 12000    # the size from which masks are scanned
    g = sva.make_geometry(H, d, F, Hp, Wp, num_slots=W + n, pairs=rope_pairs_for(d), max_frames=F * (W + 3))
    cache = sva.Cache(g)
    gen = torch.Generator(device="cuda").manual_seed(11)
    draw = lambda: torch.randn((1, T, H, d), generator=gen, device="cuda").bfloat16()  # noqa: E731
    ctx, entries = [], []
    for j in range(W):
        s = cache.bind(0, W - j, 0)
        cache.rope_kv_write([dict(seq=0, chunk=W - j, level=0, own_slot=s)], draw(), draw())
        ctx.append(s)
    for i in range(n):
        s = cache.bind(0, W + 1, i)
        cache.rope_kv_write([dict(seq=0, chunk=W + 1, level=i, own_slot=s)], draw(), draw())
        entries.append(dict(seq=0, chunk=W + 1, level=i, own_slot=s, ctx=ctx[:W - i],
                            visible=f.get("visible", [1] * W)[:W - i], within=int(f.get("causal", False))))
    nodes = sva.make_nodes(entries)
    q = torch.cat([draw() for _ in range(n)])

    # blocks of 100 queries x 200 keys, one in four kept, one state wholly hidden, junk past T
    def words(states, extra):
        m = torch.rand((n, T // 100, states, T // 200 + 1), generator=gen, device="cuda") < 0.25
        m = m.repeat_interleave(100, 1).repeat_interleave(200, 3)[..., :T]
        m[:, :, states - 1] = False
        m[:, 300:420] = False                       # a run of queries across a tile edge that see nothing
        full = torch.ones(m.shape[:-1] + (-(-T // 32) * 32 + 32 * extra,), dtype=torch.bool, device="cuda")
        full[..., :T] = m
        return pack_bits(full.cpu(), full.shape[-1] // 32).cuda()

    extra, states = f.get("extra", 0), f.get("states", W)
    own = words(2, extra)[:, :, 0].contiguous() if f.get("own", True) else None
    hist = words(states, extra) if f.get("hist", True) else None
    tile = None
    if f.get("tiles"):
        keep = torch.rand((n, nt, (1 + W) * nt), generator=gen, device="cuda") < 0.7
        tile = pack_bits(keep.cpu(), -(-(1 + W) * nt // 32)).cuda()
    got = []
    for ws in (False, True):
        if ws:
            buf = torch.full((cache.workspace_bytes(),), 255, dtype=torch.uint8, device="cuda")
            cache.set_workspace(buf)
        for _ in range(2):     # the second call finds the first one's bytes in the workspace
            out = torch.full_like(q, float("nan"))
            lse = torch.full((n, H, T), float("nan"), device="cuda")
            cache.attend_nodes_masked(nodes, q, out, lse, tile_mask=tile, own_mask=own, hist_mask=hist)
        assert cache.poll() == sva.OK
        got.append((out.double(), lse.double()))
    (a, la), (b, lb) = got
    none = la == -math.inf
    assert torch.equal(none, lb == -math.inf)
    assert ((la - lb)[~none].abs() <= 1e-3).all()
    assert not a.isnan().any() and not b.isnan().any()
    # the results' roundings, and P's in either path: at most 2^-8 E_p|V| <= 2^-8 max |V|
    v_max = float(cache.slot_pool()[:, 1].abs().max())
    assert ((a - b).abs() <= 2.0 ** -8 * (a.abs() + b.abs()) + 2 * 2.0 ** -8 * v_max).all()
    assert float((a - b).norm() / b.norm()) <= 5e-3
    cache.close()


# Masks whose rows all see every full key tile, so that a warp of the scan has a bit in each of them
# after its first rows, and whose ragged last tile only the last rows of every query tile see: it may
# not be given up before all rows are read.  With `rare` a full tile is seen by one row in 256 as
# well.  T leaves 1 to 4 words in the last tile, or has more words than one pass over a row takes
# (256).  The keys of those tiles are large, so that a row which lost them is off by far more than
# the bound.
@pytest.mark.parametrize("rare", [False, True])
@pytest.mark.parametrize("which", ["own", "history"])
@pytest.mark.parametrize("T,H,W", [(2580, 12, 4), (2610, 12, 4), (2500, 12, 4), (2680, 12, 4), (2560, 12, 4),
                                   (8220, 4, 1)])
def test_scan_reads_every_row(T, H, W, which, rare):
    d, nt, words = 64, -(-T // 128), -(-T // 32)
    assert H * -(-nt // 2) * (W + 1) * nt >= 12000    # the size from which masks are scanned
    cache = sva.Cache(sva.make_geometry(H, d, 1, 1, T, num_slots=W + 1, pairs=rope_pairs_for(d), max_frames=W + 4))
    gen = torch.Generator(device="cuda").manual_seed(T)
    draw = lambda: torch.randn((1, T, H, d), generator=gen, device="cuda")  # noqa: E731
    last, few = (nt - 1) * 128, 3 * 128      # first keys of the last tile and of the rarely seen one
    slots = []
    for b in range(W + 1, 0, -1):
        k = draw()
        k[0, last:] *= 40.0
        k[0, few:few + 128] *= 40.0
        s = cache.bind(0, b, 0)
        cache.rope_kv_write([dict(seq=0, chunk=b, level=0, own_slot=s)], k.bfloat16(), draw().bfloat16())
        slots.append(s)
    nodes = sva.make_nodes([dict(seq=0, chunk=W + 1, level=0, own_slot=slots[0], ctx=slots[1:])])
    q = draw().bfloat16()
    m = torch.full((1, T, words), -1, dtype=torch.int32, device="cuda")
    u = torch.arange(T, device="cuda")
    m[0, :, last // 32:][(u % 128 < 110) & (u < T - 5)] = 0
    if rare:
        m[0, :, few // 32:few // 32 + 4][u % 256 != 255] = 0
    own = m if which == "own" else None
    hist = m[:, :, None].repeat(1, 1, W, 1) if which == "history" else None
    got = []
    for ws in (False, True):
        if ws:
            cache.set_workspace(torch.empty(cache.workspace_bytes(), dtype=torch.uint8, device="cuda"))
        out, lse = torch.empty_like(q), torch.empty((1, H, T), device="cuda")
        cache.attend_nodes_masked(nodes, q, out, lse, own_mask=own, hist_mask=hist)
        assert cache.poll() == sva.OK
        got.append((out.double(), lse.double()))
    (a, la), (b, lb) = got
    # the same logits in either path; the fp32 sums over the keys in another order
    assert ((la - lb).abs() <= 1e-3 + 2.0 ** -20 * la.abs()).all()
    v_max = float(cache.slot_pool()[:, 1].abs().max())
    assert ((a - b).abs() <= 2.0 ** -8 * (a.abs() + b.abs()) + 2 * 2.0 ** -8 * v_max).all()
    cache.close()
