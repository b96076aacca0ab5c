"""Failure detection without a GPU fault: the test hook makes one K/V copy
never arrive, the kernel's bounded wait expires after 0.2 s, every CTA
records SVA_ERR_DEVICE_TIMEOUT, drains and exits, and the host reads the
status.  The context stays usable: the next launch succeeds and reproduces
the earlier output bit for bit."""
import pytest
import torch

from paper_2609_22283_gb300 import inputs as I
from tests import _parity as P

pytestmark = pytest.mark.gpu


def test_bounded_wait_reports_timeout(sva_mod):
    sva = sva_mod
    w = I.WORKLOADS["tiny"]
    inp = I.generate(w)
    step, q, out, lse = P.gpu_step(w, inp)
    nodes, n = step.node_table()
    c = step.cache
    before = out.clone()
    junk = torch.empty_like(out)
    c.debug_inject(1, 0.2)
    c.attend_nodes(nodes, q, junk, None, step.scale, check=False)
    assert c.poll() == sva.ERR_DEVICE_TIMEOUT
    assert "bounded wait" in sva.last_error()
    assert c.poll() == sva.OK                      # the status word was cleared
    c.debug_inject(0, 1.0)
    again = torch.empty_like(out)
    c.attend_nodes(nodes, q, again, None, step.scale, check=False)
    assert c.poll() == sva.OK
    assert torch.equal(again.view(torch.int16), before.view(torch.int16))
    step.close()


@pytest.mark.parametrize("d", [64, 128])
def test_timeout_in_one_range_of_a_cluster(sva_mod, d):
    """A unit of six key tiles is split over a cluster of three CTAs; a tile
    mask leaves four tiles, one for each of the first two CTAs and two for the
    last, whose second V copy the hook withholds.  Only that CTA times out: the
    others must not merge what never arrived, so nothing of the unit is
    written."""
    sva = sva_mod
    T, W, H = 256, 2, 2
    c = sva.Cache(sva.make_geometry(H, d, 1, 1, T, num_slots=W + 1, pairs=I.rope_pairs_for(d), max_frames=W + 3))
    c.set_workspace(torch.empty(c.workspace_bytes(), dtype=torch.uint8, device="cuda"))
    gen = torch.Generator(device="cuda").manual_seed(d)
    draw = lambda: torch.randn((1, T, H, d), generator=gen, device="cuda").bfloat16()  # noqa: E731
    slots = []
    for b in range(W + 1, 0, -1):
        slots.append(c.bind(0, b, 0))
        c.rope_kv_write([dict(seq=0, chunk=b, level=0, own_slot=slots[-1])], draw(), draw())
    nodes = sva.make_nodes([dict(seq=0, chunk=W + 1, level=0, own_slot=slots[0], ctx=slots[1:])])
    q = draw()
    mask = torch.full((1, 2, 1), 0b110101, dtype=torch.int32, device="cuda")
    before = torch.empty_like(q)
    c.attend_nodes_sparse(nodes, q, before, mask)
    assert c.poll() == sva.OK
    out, lse = torch.full_like(q, 7.0), torch.full((1, H, T), 7.0, device="cuda")
    c.debug_inject(1, 0.2)
    c.attend_nodes_sparse(nodes, q, out, mask, lse)
    assert c.poll() == sva.ERR_DEVICE_TIMEOUT
    assert bool((out == 7.0).all()) and bool((lse == 7.0).all())
    c.debug_inject(0, 1.0)
    c.attend_nodes_sparse(nodes, q, out, mask, lse)
    assert c.poll() == sva.OK
    assert torch.equal(out, before)
    c.close()
