"""Backward pass with lists of streamed rows cut over clusters of CTAs: items of one row and of full tiles,
ragged blocks, both head dims, batches; against the oracle's derivative, twice bit for bit, and in a row with
the next call (its statistics pass must not overtake this call's launches)."""
import numpy as np
import pytest
import torch

from oracle import attn_c
from oracle import hilberta_oracle as orc
from paper_2509_26538_b200 import binding as hb

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,W,tile,o,hs,nt,B,heads,D", [
    (16, 32, 256, 100, 2, 20, 1, 1, 128),     # few units, but too short to be cut
    (32, 32, 256, 128, 4, 64, 1, 8, 128),     # prefix items cut, window items not
    (32, 32, 256, 128, 4, 64, 1, 8, 64),
    (48, 40, 1024, 77, 8, 226, 1, 2, 128),    # prefix of two full tiles and a rest
    (48, 40, 1024, 77, 8, 226, 3, 3, 64),
    (48, 48, 4096, 0, 0, 1, 1, 1, 128),   # one dense tile and one token more
    (64, 64, 512, 0, 8, 512, 1, 3, 128),
])
def test_matches_the_derivative(H, W, tile, o, hs, nt, B, heads, D):
    S = nt + H * W
    g = torch.Generator().manual_seed(S + D + heads)
    q, k, v, do = (torch.randn((B, heads, S, D), generator=g).to(torch.bfloat16) for _ in range(4))
    ig, grp = orc.token_classes(H, W, tile, o, hs, nt)
    refs = attn_c.attention_backward(q.float().numpy(), k.float().numpy(), v.float().numpy(), do.float().numpy(), ig, grp)
    plan = hb.Plan(H, W, tile, o, hs, nt)
    dev = [t.cuda() for t in (q, k, v, do)]
    p = [torch.empty_like(t) for t in dev]
    for src, dst in zip(dev, p):
        plan.permute(src, dst)
    plan.bind_like(p[0])
    out, lse = torch.empty_like(p[0]), torch.empty((B, heads, S), device="cuda")
    plan.forward_lse(p[0], p[1], p[2], out, lse)
    runs = [[torch.full_like(out, float("nan")) for _ in range(3)] for _ in range(3)]
    other = [torch.empty_like(out) for _ in range(3)]
    plan.backward(p[3], p[0], p[1], p[2], out, lse, *runs[0])
    plan.backward(p[0], p[1], p[2], p[3], out, lse * 0 + 9, *other)   # other inputs, other statistics, right behind
    plan.backward(p[3], p[0], p[1], p[2], out, lse, *runs[1])
    plan.backward(p[3], p[0], p[1], p[2], out, lse, *runs[2])
    assert plan.status() == 0
    for a, b, c in zip(*runs):
        assert torch.equal(a.view(torch.int16), b.view(torch.int16)) and torch.equal(a.view(torch.int16), c.view(torch.int16))
    back = torch.empty_like(out)
    for t, r in zip(runs[0], refs):
        plan.unpermute(t, back)
        got = back.cpu().double().numpy()
        assert orc.rel_l2_err(got, r) <= 5e-3
        assert np.abs(got - r).max() <= 1e-2 * max(1.0, np.abs(r).max())
    plan.destroy()
