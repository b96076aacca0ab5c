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
|d| <= 2^-8 (E_p|V| + |O|) + 2^-9 E_p|V|."""
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
    bound = 2.0 ** -8 * (ev + o.abs()) + 2.0 ** -9 * ev
    bad = ~((out[0].double() - o).abs() <= bound)
    assert not bad.any(), f"{int(bad.sum())} of {bad.numel()} elements out of bound"
    ref = torch.logsumexp(s, dim=-1)
    none = ref == -math.inf
    assert (lse[0][none] == -math.inf).all()
    assert ((lse[0].double() - ref)[~none].abs() <= 2e-3 + 2.0 ** -20 * ref[~none].abs()).all()
    cache.close()
