"""Small attention launches where the loop and the splits can go wrong: one and
two query tiles, key-tile counts around the lengths of the S, K and V rings (at
d = 64: 3, 4 and 6), a query-tile pair whose second tile is missing, unsplit
and (with a workspace) split over clusters of two to eight CTAs, and keys whose
size grows from state to state, so that the running max jumps past the lazy
rescale threshold in mid-sequence.

Reference: the same op in fp64 torch on the rotated Q and the K', V the cache
holds.  Bound per element: the rounding of P to bf16 moves O by at most
2^-8 E_p|V|, that of the output by at most 2^-8 |O|, and fp32 logits of size
L carry an error of about 2^-22 L (L < 2^11 log2 units here, so 2^-11), which
scales the weights: |d| <= 2^-8 (E_p|V| + |O|) + 2^-10 E_p|V|, and 2^-20 for
the fp32 sums themselves (|V| < 8), which is all that is left where a row's
whole weight sits on a key whose V is about zero."""
import math

import pytest
import torch

from paper_2609_22283_gb300 import sva
from paper_2609_22283_gb300.inputs import rope_pairs_for

pytestmark = pytest.mark.gpu


def _reference(cache, node, q, i, scale):
    """(O, E_p|V|, lse) of node i, [T][H][d] and [H][T], in fp64."""
    pool, T = cache.slot_pool(), cache.T
    slots = [node.own_slot] + [node.ctx_slot[j] for j in range(node.n_ctx)]
    k = torch.cat([pool[s, 0, :, :T] for s in slots], dim=1).double()
    v = torch.cat([pool[s, 1, :, :T] for s in slots], dim=1).double()
    s = torch.einsum("thd,hkd->htk", q[i].double(), k) * scale
    p = torch.softmax(s, dim=-1)
    return (torch.einsum("htk,hkd->thd", p, v), torch.einsum("htk,hkd->thd", p, v.abs()),
            torch.logsumexp(s, dim=-1))


@pytest.mark.parametrize("split", [False, True])
@pytest.mark.parametrize("grow", [1.0, 20.0])
@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("T,W", [(128, 0), (100, 2), (130, 0), (200, 1), (256, 3), (300, 2), (257, 6),
                                 (120, 6), (250, 4), (250, 5), (90, 15)])
def test_small_launches(T, W, d, grow, split):
    H, n = 2, 2
    g = sva.make_geometry(H, d, 1, 1, T, num_slots=W + n, pairs=rope_pairs_for(d), max_frames=W + 4)
    cache = sva.Cache(g)
    if split:
        cache.set_workspace(torch.empty(cache.workspace_bytes(), dtype=torch.uint8, device="cuda"))
    gen = torch.Generator().manual_seed(T * 31 + W)
    draw = lambda by=1.0: (torch.randn((1, T, H, d), generator=gen) * by).bfloat16().cuda()  # noqa: E731
    ctx, entries = [], []
    for j in range(W):   # the walk goes from the newest state to the oldest: the oldest has the largest keys
        s = cache.bind(0, W - j, 0)
        cache.rope_kv_write([dict(seq=0, chunk=W - j, level=0, own_slot=s)], draw(grow * (j + 1)), draw())
        ctx.append(s)
    for i in range(n):
        s = cache.bind(0, W + 1, i)
        cache.rope_kv_write([dict(seq=0, chunk=W + 1, level=i, own_slot=s)], draw(), draw())
        entries.append(dict(seq=0, chunk=W + 1, level=i, own_slot=s, ctx=ctx))
    nodes = sva.make_nodes(entries)
    q = torch.cat([draw() for _ in range(n)])
    out, lse = torch.empty_like(q), torch.empty((n, H, T), dtype=torch.float32, device="cuda")
    cache.attend_nodes(nodes, q, out, lse)
    assert cache.poll() == sva.OK
    for i in range(n):
        o, ev, l = _reference(cache, nodes[i], q, i, 1.0 / math.sqrt(d))
        bound = 2.0 ** -8 * (ev + o.abs()) + 2.0 ** -10 * ev + 2.0 ** -20
        bad = (out[i].double() - o).abs() > bound
        assert not bad.any(), f"node {i}: {int(bad.sum())} of {bad.numel()} elements out of bound"
        assert (lse[i].double() - l).abs().max() <= 2e-3 + 2.0 ** -20 * l.abs().max()
    cache.close()
