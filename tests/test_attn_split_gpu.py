"""Tensor-core forward with long key lists cut over clusters of CTAs: every way in and out (physical and
original order, log-sum-exp, fp8, head dim 64), items of one and of two query tiles, ragged last blocks,
batches, more heads than clusters.  Bars as for the uncut kernels; the same launch twice is bit-identical."""
import numpy as np
import pytest
import torch

from oracle import attn_c
from oracle import hilberta_oracle as orc
from paper_2509_26538_b200 import binding as hb

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,W,tile,o,hs,nt,B,heads,D,fp8", [
    (16, 32, 256, 100, 2, 20, 1, 1, 128, False),    # few units, but too short to be cut
    (32, 32, 256, 128, 4, 64, 1, 8, 128, False),    # one-tile prefix items beside uncut window items
    (32, 32, 256, 128, 4, 64, 1, 8, 64, False),
    (32, 32, 256, 128, 4, 64, 1, 8, 128, True),
    (48, 40, 1024, 77, 8, 226, 1, 2, 128, False),   # prefix of two full tiles and a rest, ragged blocks
    (48, 40, 1024, 77, 8, 226, 1, 2, 128, True),
    (48, 40, 1024, 77, 8, 226, 3, 5, 64, False),
    (64, 64, 512, 0, 8, 512, 1, 3, 128, False),
    (64, 64, 4096, 0, 0, 1, 1, 1, 128, False),      # one dense tile
])
def test_every_way_through(H, W, tile, o, hs, nt, B, heads, D, fp8):
    S = nt + H * W
    g = torch.Generator().manual_seed(S + D + heads)
    dt = torch.float8_e4m3fn if fp8 else torch.bfloat16
    q, k, v = (torch.randn((B, heads, S, D), generator=g).to(dt) for _ in range(3))
    ig, grp = orc.token_classes(H, W, tile, o, hs, nt)
    ref, ref_lse = attn_c.attention_rows(q.float().numpy(), k.float().numpy(), v.float().numpy(), ig, grp, return_lse=True)
    bars = (2 ** -4 * float(v.float().abs().max()) + 1e-2, 4e-2) if fp8 else (1e-2, 5e-3)
    plan = hb.Plan(H, W, tile, o, hs, nt)
    qd, kd, vd = (t.cuda() for t in (q, k, v))
    qp, kp, vp = (torch.empty_like(qd) for _ in range(3))
    for src, dst in ((qd, qp), (kd, kp), (vd, vp)):
        plan.permute(src, dst)
    plan.bind_like(qp)
    outs = [torch.full((B, heads, S, D), float("nan"), dtype=torch.bfloat16, device="cuda") for _ in range(5)]
    lse = torch.full((B, heads, S), float("nan"), device="cuda")
    plan.forward(qp, kp, vp, outs[0])
    plan.forward_lse(qp, kp, vp, outs[1], lse)
    plan.forward_unpermute(qp, kp, vp, outs[2])
    plan.forward_fused(qd, kd, vd, outs[3])
    plan.unpermute(outs[0], outs[4])
    assert plan.status() == 0
    bits = [t.view(torch.int16) for t in outs]
    assert torch.equal(bits[0], bits[1])
    assert torch.equal(bits[2], bits[4]) and torch.equal(bits[3], bits[4])
    got = outs[4].cpu().double().numpy()
    assert orc.max_abs_err(got, ref) <= bars[0] and orc.rel_l2_err(got, ref) <= bars[1]
    order = plan.export(hb.EXPORT_PHYS2ORIG)
    assert np.abs(lse.cpu().double().numpy() - ref_lse[:, :, order]).max() <= 2e-3
    host = torch.full((B, heads, S, D), float("nan"), dtype=torch.bfloat16)
    plan.forward_host(q, k, v, host)
    assert torch.equal(host.view(torch.int16), bits[4].cpu())
    plan.destroy()


def test_two_streams_share_a_plan():
    """Launches of one plan on two streams at once: the merge keeps nothing outside the launch."""
    H = W = 64
    plan = hb.Plan(H, W, 512, 100, 8, 300)
    S = 300 + H * W
    g = torch.Generator().manual_seed(5)
    sets = [[torch.randn((1, 2, S, 128), generator=g).to(torch.bfloat16).cuda() for _ in range(3)] for _ in range(2)]
    plan.bind_like(sets[0][0])
    want = [plan.forward(*s, torch.empty_like(s[0])) for s in sets]
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream() for _ in range(2)]
    got = [[torch.empty_like(s[0]) for _ in range(20)] for s in sets]
    for i in range(20):
        for s, st, out in zip(sets, streams, got):
            plan.forward(*s, out[i], stream=st)
    torch.cuda.synchronize()
    assert plan.status() == 0
    for w, outs in zip(want, got):
        assert all(torch.equal(w.view(torch.int16), t.view(torch.int16)) for t in outs)
    plan.destroy()


@pytest.mark.parametrize("D,fp8", [(128, False), (64, False), (128, True)])
def test_values_that_are_not_finite(D, fp8):
    """Keys of the first half score far below those of the second, so that their share of the weight is exactly zero:
    a NaN among their values is in the result all the same, and scores of -inf there are not."""
    H = W = 64
    plan = hb.Plan(H, W, 512, 0, 8, 512)
    S, P, heads = plan.S, 512 + 64, 3
    g = torch.Generator(device="cuda")
    g.manual_seed(2)
    dt = torch.float8_e4m3fn if fp8 else torch.bfloat16
    d = torch.randn(D, generator=g, device="cuda").sign()
    q = (12 * d).expand(1, heads, S, D).contiguous()
    k = torch.where(torch.arange(S, device="cuda")[:, None] < S // 2, -12 * d, 12 * d).expand(1, heads, S, D).contiguous()
    v = torch.randn((1, heads, S, D), generator=g, device="cuda")
    q, k, v = q.to(dt), k.to(dt), v.to(dt)
    plan.bind_like(q)
    out = torch.empty((1, heads, S, D), dtype=torch.bfloat16, device="cuda")
    plan.forward(q, k, v, out)
    want = v[:, :, S // 2:].double().mean(2, keepdim=True)   # the second half's keys weigh the same
    assert (out[:, :, :P].double() - want).abs().max() <= 2 ** -6
    for at in (0, 600, S // 2 - 1, S - 1):
        bad = v.clone()
        bad.view(torch.uint8 if fp8 else torch.int16)[0, 1, at, 5] = 0x7f if fp8 else 0x7fc0
        plan.forward(q, k, bad, out)
        assert torch.isnan(out[0, 1, :P, 5].float()).all(), at
        assert torch.isfinite(out[0, 0, :P].float()).all() and torch.isfinite(out[0, 2, :P].float()).all()
    if not fp8:   # finite keys whose scores overflow
        k[:, :, S // 2:] = 0   # the others score 0
        k[:, :, S - 200:S - 100] = (-3e38 * d).to(dt)
        plan.forward(q, k, v, out)
        assert torch.isfinite(out[:, :, :P].float()).all()
    assert plan.status() == 0
    plan.destroy()
