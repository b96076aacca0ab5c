"""The RMSNorm + RoPE + cache write at the row widths where its kernel changes
shape (one to eight warps a token, two to eight 16-byte vectors a lane), with
token counts that leave part of the last block idle, with and without queries;
and at the token counts, relative to the GPU's SMs, where it is given to the
kernel that reads its rows twice, or just is not.

Against fp64 torch: the result is rounded to bf16 once (2^-8 relative) after
fp32 arithmetic, whose error is a few 2^-24 of the rotated pair's length (16
of them here: sum of squares, reciprocal square root, two products and the
rotation), so |d| <= 2^-8 |ref| + 2^-20 |pair|."""
import pytest
import torch

from paper_2609_22283_gb300 import sva
from paper_2609_22283_gb300.inputs import rope_pairs_for

pytestmark = pytest.mark.gpu


def _reference(x, gamma, t0, T, Wp, d, eps):
    """[T][H][d] normalised over H*d and rotated, fp64; and each element's pair length."""
    y = x.double().reshape(T, -1)
    y = (y * torch.rsqrt((y * y).mean(1, keepdim=True) + eps) * gamma.double()).reshape(x.shape)
    u = torch.arange(T, device=x.device)
    ang = []
    for pos, p in zip((torch.full_like(u, t0), u // Wp, u % Wp), rope_pairs_for(d)):
        ang.append(pos.double()[:, None] * 10000.0 ** (-torch.arange(p, device=x.device).double() / p))
    a = torch.cat(ang, 1)[:, None]
    y = y.reshape(T, -1, d // 2, 2)
    out = torch.stack((y[..., 0] * a.cos() - y[..., 1] * a.sin(), y[..., 0] * a.sin() + y[..., 1] * a.cos()), -1)
    return out.reshape(x.shape), y.norm(dim=-1, keepdim=True).expand_as(y).reshape(x.shape)


@pytest.mark.parametrize("with_q", [False, True])
@pytest.mark.parametrize("H,d", [(1, 64), (8, 64), (9, 64), (12, 128), (13, 128), (24, 128), (25, 128), (32, 128),
                                 (33, 128), (40, 128), (41, 128), (48, 128), (128, 64), (80, 128), (81, 128),
                                 (128, 128)])
def test_norm_widths(H, d, with_q):
    _check(H, d, with_q, 3, 15)


# tokens per SM: just inside and just past the ranges in which the launch takes the other kernel
@pytest.mark.parametrize("with_q", [False, True])
@pytest.mark.parametrize("H,d", [(17, 64), (16, 128), (28, 128), (48, 128)])
@pytest.mark.parametrize("per_sm,past", [(8, True), (12, True), (16, False), (16, True), (24, True), (32, False),
                                         (32, True)])
def test_norm_token_counts(per_sm, past, H, d, with_q):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    _check(H, d, with_q, 1, per_sm * sms // 3 + past, device="cuda")


def _check(H, d, with_q, Hp, Wp, device="cpu"):
    n, eps = 3, 1e-6
    T = Hp * Wp
    cache = sva.Cache(sva.make_geometry(H, d, 1, Hp, Wp, num_slots=n, pairs=rope_pairs_for(d), max_frames=16))
    gen = torch.Generator(device=device).manual_seed(H * 1000 + d)
    draw = lambda: (torch.randn((n, T, H, d), generator=gen, device=device) * 3).bfloat16().cuda()  # noqa: E731
    k, v, q = draw(), draw(), draw()
    gk, gq = (torch.rand(H * d, generator=gen, device=device).cuda() + 0.5 for _ in range(2))
    chunks = [2, 7, 11]
    slots = [cache.bind(0, c, 1) for c in chunks]
    nodes = [dict(seq=0, chunk=c, level=1, own_slot=s) for c, s in zip(chunks, slots)]
    q0, pads = q.clone(), cache.slot_pool()[:, :, :, T:].clone()
    cache.rope_kv_write_qknorm(nodes, k, v, q if with_q else None, gk, gq if with_q else None, eps)
    assert cache.poll() == sva.OK
    pool = cache.slot_pool()
    for i, (c, s) in enumerate(zip(chunks, slots)):
        assert torch.equal(pool[s, 1, :, :T].transpose(0, 1), v[i])
        got = [(pool[s, 0, :, :T].transpose(0, 1), k[i], gk)] + ([(q[i], q0[i], gq)] if with_q else [])
        for y, x, g in got:
            ref, pair = _reference(x, g, c, T, Wp, d, eps)
            assert ((y.double() - ref).abs() <= 2.0 ** -8 * ref.abs() + 2.0 ** -20 * pair).all()
    assert torch.equal(pool[:, :, :, T:], pads) and (with_q or torch.equal(q, q0))
    cache.close()
