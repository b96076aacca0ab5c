"""Key ranges merged through the workspace: launches of a few more units than
SMs, whose full wave runs unsplit and whose last units are split four ways
(small launches are merged inside clusters instead), dense, with a tile mask
that leaves some ranges nothing, with token masks, and under frame causality
with a range that some rows see nothing of.  The workspace is filled with ones
first, so that the partials written there show how many ranges there were.

Reference: the same op in fp64 torch on the rotated Q and the K', V the cache
holds.  Bound as for other small launches: the rounding of P moves O by at most
2^-8 E_p|V|, that of the output by 2^-8 |O|, and fp32 logits below 2^11 log2
units carry an error of about 2^-11, which scales the weights: |d| <=
2^-8 (E_p|V| + |O|) + 2^-10 E_p|V|, and 2^-20 for the fp32 sums."""
import math

import pytest
import torch

from paper_2609_22283_gb300 import sva
from paper_2609_22283_gb300.inputs import pack_bits, rope_pairs_for

pytestmark = pytest.mark.gpu


class Launch:
    def __init__(self, F, Hp, Wp, H, d, n, W, grow=1.0, causal=False):
        self.T, self.H, self.d, self.n, self.W, self.fr = F * Hp * Wp, H, d, n, W, Hp * Wp
        self.causal = causal
        self.c = sva.Cache(sva.make_geometry(H, d, F, Hp, Wp, num_slots=W + n, pairs=rope_pairs_for(d),
                                             max_frames=F * (W + 3)))
        self.ws = torch.full((self.c.workspace_bytes(),), 255, dtype=torch.uint8, device="cuda")
        self.c.set_workspace(self.ws)
        gen = torch.Generator(device="cuda").manual_seed(d + W)
        draw = lambda by=1.0: (torch.randn((1, self.T, H, d), generator=gen, device="cuda") * by).bfloat16()  # noqa: E731
        self.ctx, entries = [], []
        for j in range(W):
            s = self.c.bind(0, W - j, 0)
            self.c.rope_kv_write([dict(seq=0, chunk=W - j, level=0, own_slot=s)], draw(grow * (j + 1)), draw())
            self.ctx.append(s)
        for i in range(n):
            s = self.c.bind(0, W + 1, i)
            self.c.rope_kv_write([dict(seq=0, chunk=W + 1, level=i, own_slot=s)], draw(), draw())
            entries.append(dict(seq=0, chunk=W + 1, level=i, own_slot=s, ctx=self.ctx, within=int(causal)))
        self.own = [e["own_slot"] for e in entries]
        self.nodes = sva.make_nodes(entries)
        self.q = torch.cat([draw() for _ in range(n)])

    def run(self, ranges, **masks):
        """Two calls, the same bits; `ranges` partials in the workspace, the counters at zero."""
        got = []
        for _ in range(2):
            out = torch.full_like(self.q, float("nan"))
            lse = torch.full((self.n, self.H, self.T), float("nan"), device="cuda")
            self.c.attend_nodes_masked(self.nodes, self.q, out, lse, **masks)
            assert self.c.poll() == sva.OK
            got.append((out, lse))
        assert torch.equal(got[0][0], got[1][0]) and torch.equal(got[0][1], got[1][1])
        sms = torch.cuda.get_device_properties(0).multi_processor_count
        counters = -(-4 * sms * 4 // 256) * 256
        assert not self.ws[:counters].any()
        items = self.ws[counters:].view(torch.int32).view(4 * sms, 256 * (self.d + 2))
        written = items[:, 256 * self.d] != -1      # the first row's maximum
        assert int(written.sum()) == ranges and bool(written[:ranges].all())
        return got[0]

    def check(self, out, lse, see, heads):
        """see: bool [n][T][(1 + W) T], the visible keys."""
        pool, T = self.c.slot_pool(), self.T
        for i in range(self.n):
            slots = [self.own[i]] + self.ctx
            for h in heads:
                k, v = (torch.cat([pool[s, kv, h, :T] for s in slots]).double() for kv in (0, 1))
                s = self.q[i, :, h].double() @ k.T / math.sqrt(self.d)
                s.masked_fill_(~see[i], -math.inf)
                p = torch.nan_to_num(torch.softmax(s, dim=-1), nan=0.0)
                o, ev = p @ v, p @ v.abs()
                bound = 2.0 ** -8 * (ev + o.abs()) + 2.0 ** -10 * ev + 2.0 ** -20
                bad = ~((out[i, :, h].double() - o).abs() <= bound)
                assert not bad.any(), f"node {i} head {h}: {int(bad.sum())} of {bad.numel()} elements out of bound"
                l = torch.logsumexp(s, dim=-1)
                none = l == -math.inf
                assert (lse[i, h][none] == -math.inf).all()
                assert ((lse[i, h].double() - l)[~none].abs() <= 2e-3 + 2.0 ** -20 * l[~none].abs()).all()


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("form", ["dense", "tiles", "tokens", "tiles and tokens"])
def test_four_way_merge(form, d):
    n, W = 2, 7
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    units = sms + 8 + sms % 2
    a = Launch(1, 8, 30, units // n, d, n, W, grow=5.0)
    T, nt, S = a.T, 2, 1 + W
    gen = torch.Generator().manual_seed(3)
    see = torch.ones((n, T, S, T), dtype=torch.bool)
    masks = {}
    if "tiles" in form:
        keep = torch.rand((n, nt, S * nt), generator=gen) < 0.5
        keep[1] = False
        keep[1, 0, 3], keep[1, 1, 8], keep[1, :, 15] = True, True, True   # three tiles for four ranges
        masks["tile_mask"] = pack_bits(keep, 1).cuda()
        rows = keep.repeat_interleave(128, 1)[:, :T].view(n, T, S, nt)
        see &= rows.repeat_interleave(128, 3)[..., :T]
    if "tokens" in form:
        m = torch.rand((n, T, S, T), generator=gen) < 0.4
        m[:, 17] = False                       # a query that sees nothing
        m[:, 40:60, 2:6] = False               # queries whose middle ranges are empty
        masks["own_mask"] = pack_bits(m[:, :, 0], 8).cuda()
        masks["hist_mask"] = pack_bits(m[:, :, 1:], 8).cuda()
        see &= m
    out, lse = a.run(4 * (units - sms), **masks)
    a.check(out, lse, see.view(n, T, S * T).cuda(), [0, a.H // 2, a.H - 4, a.H - 1])
    a.c.close()


def test_two_way_merge_frame_causal():
    """No history, two frames of 1100 tokens: the pair of query tiles at rows 1024 to 1279 walks 18 key
    tiles in two ranges, the second of which (keys from 1152) its rows before 1100 see nothing of."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    if sms != 152:
        pytest.skip("the heads are chosen for 152 SMs")
    a = Launch(2, 22, 50, 29, 128, 2, 0, causal=True)     # 522 units: three waves and 66 units
    out, lse = a.run(132)
    frame = torch.arange(a.T, device="cuda") // a.fr
    a.check(out, lse, (frame[None, :] <= frame[:, None]).expand(2, -1, -1), [0, 25, 26, 28])
    a.c.close()


@pytest.mark.parametrize("d", [64, 128])
def test_equal_cost_goes_to_clusters(d):
    """48 units of 24 key tiles: three ranges through the workspace and clusters of two cost the plan the
    same, and clusters leave the workspace alone."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    if sms != 152:
        pytest.skip("the units are chosen for 152 SMs")
    a = Launch(1, 16, 16, 24, d, 2, 11, grow=5.0)
    out, lse = a.run(0)
    a.check(out, lse, torch.ones((2, a.T, 12 * a.T), dtype=torch.bool, device="cuda"), [0, 11, 23])
    a.c.close()
