"""Kernels of the library start while the kernel before them in the stream
still runs and wait for it on the device.  Chains of dependent calls (each
output the next one's input, cache slots, workspace counters and Q rotated in
place among them), issued without a pause, recorded in a CUDA graph, on two
streams with a cache each, and with the caller's own kernels between them,
give the bits of the same calls with a synchronisation after each."""
import pytest
import torch

from paper_2609_22283_gb300 import sva
from paper_2609_22283_gb300.inputs import pack_bits, rope_pairs_for

pytestmark = pytest.mark.gpu


class Chain:
    """A layer whose output is its next input; `between` runs after each call."""

    def __init__(self, T, H, d, W, seed, norm, masked=False):
        self.T, self.N, self.norm, self.eps = T, H * d, norm, 1e-6
        g = sva.make_geometry(H, d, 1, 1, T, num_slots=W + 1, pairs=rope_pairs_for(d), max_frames=W + 3)
        self.c = sva.Cache(g)
        self.c.set_workspace(torch.empty(self.c.workspace_bytes(), dtype=torch.uint8, device="cuda"))
        gen = torch.Generator(device="cuda").manual_seed(seed)
        draw = lambda *s, by=1.0: (torch.randn(s, generator=gen, device="cuda") * by).bfloat16()  # noqa: E731
        ctx = []
        for j in range(W):
            s = self.c.bind(0, j + 1, 0)
            self.c.rope_kv_write([dict(seq=0, chunk=j + 1, level=0, own_slot=s)], draw(1, T, H, d), draw(1, T, H, d))
            ctx.append(s)
        own = self.c.bind(0, W + 1, 0)
        self.nodes = sva.make_nodes([dict(seq=0, chunk=W + 1, level=0, own_slot=own, ctx=ctx)])
        self.w, self.b = draw(3 * self.N, self.N, by=self.N ** -0.5), torch.randn(3 * self.N, generator=gen, device="cuda")
        self.gk, self.gq = (torch.rand(self.N, generator=gen, device="cuda") + 0.5 for _ in range(2))
        self.q, self.k, self.v = (torch.empty((1, T, H, d), dtype=torch.bfloat16, device="cuda") for _ in range(3))
        self.x0 = draw(1, T, H, d)
        self.x = self.x0.clone()
        self.mask = pack_bits(torch.rand((1, T, T)) < 0.5, -(-T // 32)).cuda() if masked else None

    def steps(self, n, between=lambda: None):
        for _ in range(n):
            x = self.x.view(1, self.T, self.N)
            if self.norm:
                self.c.qkv_project(x, self.w, self.b, self.q, self.k, self.v)
                between()
                self.c.rope_kv_write_qknorm(self.nodes, self.k, self.v, self.q, self.gk, self.gq, self.eps)
            else:
                self.c.qkv_project_rope(self.nodes, x, self.w, self.b, self.q)
            between()
            if self.mask is not None:
                self.c.attend_nodes_masked(self.nodes, self.q, self.x, own_mask=self.mask)
            else:
                self.c.attend_nodes(self.nodes, self.q, self.x)
            between()

    def reset(self):
        self.x.copy_(self.x0)


SHAPES = [dict(T=320, H=12, d=128, W=3, norm=True), dict(T=64, H=2, d=64, W=2, norm=False),
          dict(T=4680, H=12, d=128, W=1, norm=True), dict(T=2500, H=6, d=64, W=2, norm=False, masked=True)]


@pytest.mark.parametrize("shape", range(len(SHAPES)))
def test_chains_of_calls(shape):
    a = Chain(seed=shape, **SHAPES[shape])
    n = 6
    a.steps(n, torch.cuda.synchronize)
    ref = a.x.clone()
    assert ref.float().abs().max() > 0 and not ref.isnan().any()
    # without a pause
    for _ in range(3):
        a.reset()
        a.steps(n)
        assert torch.equal(a.x, ref)
    # the caller's own kernels between the calls
    t = torch.ones(1 << 20, device="cuda")
    a.reset()
    a.steps(n, lambda: t.mul_(1.0))
    assert torch.equal(a.x, ref)
    # recorded
    st = torch.cuda.Stream()
    g = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(g, stream=st):
        a.steps(n)
    for _ in range(2):
        a.reset()
        torch.cuda.synchronize()
        g.replay()
        torch.cuda.synchronize()
        assert torch.equal(a.x, ref)
    # two streams, a cache each
    b = Chain(seed=shape, **SHAPES[shape])
    if b.mask is not None:
        b.mask.copy_(a.mask)
    a.reset()
    torch.cuda.synchronize()
    s1, s2 = torch.cuda.Stream(), torch.cuda.Stream()
    for _ in range(n):
        with torch.cuda.stream(s1):
            a.steps(1)
        with torch.cuda.stream(s2):
            b.steps(1)
    torch.cuda.synchronize()
    assert torch.equal(a.x, ref) and torch.equal(b.x, ref)
    assert a.c.poll() == sva.OK and b.c.poll() == sva.OK
    a.c.close(), b.c.close()


@pytest.mark.parametrize("captured", [False, True])
@pytest.mark.parametrize("shape", [0, 1])
def test_fork_and_join(shape, captured):
    """Two chains on two streams, joined by events into one tensor that the first chain reads next."""
    a, b = Chain(seed=10, **SHAPES[shape]), Chain(seed=11, **SHAPES[shape])
    fork = torch.empty_like(a.x)        # what b reads while a goes on to overwrite a.x

    def step(main, side, wait=False):
        with torch.cuda.stream(main):
            a.steps(1)
            fork.copy_(a.x)
            side.wait_stream(main)
            if wait:
                torch.cuda.synchronize()
        with torch.cuda.stream(side):
            b.x.add_(fork)
            b.steps(1)
            if wait:
                torch.cuda.synchronize()
        with torch.cuda.stream(main):
            a.steps(1)
            main.wait_stream(side)      # our kernel next, straight after the join
            a.c.qkv_project(b.x.view(1, a.T, a.N), a.w, a.b, a.q, a.k, a.v)
            a.x.copy_(a.q)
            if wait:
                torch.cuda.synchronize()

    def run(main, side, wait=False):
        for _ in range(4):
            step(main, side, wait)

    main, side = torch.cuda.Stream(), torch.cuda.Stream()
    torch.cuda.synchronize()
    run(main, side, wait=True)
    ref = a.x.clone(), b.x.clone()
    a.reset(), b.reset()
    torch.cuda.synchronize()
    if captured:
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=main):
            run(main, side)
        a.reset(), b.reset()
        torch.cuda.synchronize()
        g.replay()
    else:
        run(main, side)
    torch.cuda.synchronize()
    assert torch.equal(a.x, ref[0]) and torch.equal(b.x, ref[1])
    a.c.close(), b.c.close()
