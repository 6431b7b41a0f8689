"""fp32 kernels where their tiling can go wrong: one block of 32 keys and its neighbours, lists cut over
clusters (more shares than blocks included), rows past a 64-row item, ranges that wrap inside a block."""
import numpy as np
import pytest
import torch

from oracle import attn_c
from oracle import hilberta_oracle as orc
from paper_2509_26538_b200 import binding as hb

pytestmark = pytest.mark.gpu

TOL = 1e-5   # the fp32 path's bar on both metrics


@pytest.mark.parametrize("H,W,tile,o,hs,nt,B,heads,D", [
    (4, 8, 64, 0, 0, 0, 1, 1, 64),        # 32 keys: exactly one block, nothing to cut
    (4, 8, 64, 0, 0, 1, 1, 1, 128),       # 33 keys: one key in the second block
    (8, 8, 64, 5, 0, 1, 1, 1, 32),        # 65 rows: one row in the second item, three blocks in eight shares
    (16, 16, 128, 100, 2, 31, 1, 2, 64),  # wrapped tiles, a prefix that ends inside a block
    (13, 29, 256, 77, 4, 50, 1, 3, 64),   # ragged everywhere, clusters of eight
    (32, 32, 256, 128, 4, 64, 1, 8, 64),  # clusters of four
    (24, 24, 256, 9, 2, 40, 2, 12, 32),   # clusters of two or none
    (16, 16, 64, 0, 2, 130, 4, 16, 128),  # many instances: no cuts
    # windows so short that their rows have a warp each
    (32, 32, 1, 0, 0, 1, 1, 8, 64),       # two keys a row: a text token and the row's own
    (32, 32, 4, 3, 0, 0, 2, 9, 32),       # no items at all, a wrapped window
    (32, 32, 16, 5, 0, 0, 1, 8, 128),     # in the backward pass only
    (24, 24, 2, 1, 2, 40, 2, 6, 64),      # beside a prefix
    (20, 27, 16, 7, 4, 33, 2, 8, 32),     # ragged: some windows short, others not, more than 32 keys a row
])
def test_forward_lse_and_backward(H, W, tile, o, hs, nt, B, heads, D):
    S = nt + H * W
    g = torch.Generator().manual_seed(H * 1000 + W + D)
    q, k, v, do = (torch.randn((B, heads, S, D), generator=g) for _ in range(4))
    ig, grp = orc.token_classes(H, W, tile, o, hs, nt)
    ref = attn_c.attention_rows(q.numpy(), k.numpy(), v.numpy(), ig, grp)
    grads = attn_c.attention_backward(q.numpy(), k.numpy(), v.numpy(), do.numpy(), ig, grp)
    plan = hb.Plan(H, W, tile, o, hs, nt)
    qd, kd, vd, dod = (t.cuda() for t in (q, k, v, do))
    # one launch with both gathers fused in
    out = torch.full_like(qd, float("nan"))
    plan.bind_like(qd)
    plan.forward_fused(qd, kd, vd, out)
    assert orc.max_abs_err(out.cpu().double().numpy(), ref) <= TOL
    assert orc.rel_l2_err(out.cpu().double().numpy(), ref) <= TOL
    # physical order: forward with log-sum-exp, backward; twice, bit for bit
    p = [torch.empty_like(qd) for _ in range(4)]
    for src, dst in zip((qd, kd, vd, dod), p):
        plan.permute(src, dst)
    runs = []
    for _ in range(2):
        op, lse = torch.full_like(qd, float("nan")), torch.full((B, heads, S), float("nan"), device="cuda")
        gp = [torch.full_like(qd, float("nan")) for _ in range(3)]
        plan.forward_lse(p[0], p[1], p[2], op, lse)
        plan.backward(p[3], p[0], p[1], p[2], op, lse, *gp)
        runs.append([op, lse] + gp)
    assert all(torch.equal(a, b) for a, b in zip(*runs))
    back = torch.empty_like(qd)
    plan.unpermute(runs[0][0], back)
    assert torch.equal(back, out)
    for t, r in zip(runs[0][2:], grads):
        plan.unpermute(t, back)
        got = back.cpu().double().numpy()
        assert orc.rel_l2_err(got, r) <= TOL
        assert np.abs(got - r).max() <= TOL * max(1.0, np.abs(r).max())
    plan.destroy()


@pytest.mark.parametrize("D", [32, 64, 128])
def test_short_windows_cost_no_more_than_long_ones(D):
    """Time, against windows of 32 tokens, which do 32 times the work: with a CTA of 64 rows for every window of one
    token the forward pass took 20 times as long and the backward pass 18."""
    H, heads = 48, 48
    g = torch.Generator(device="cuda")
    g.manual_seed(1)
    took = {}
    for tile in (1, 2, 32):
        plan = hb.Plan(H, H, tile, 0, 0, 0)
        q, k, v, do = (torch.randn((1, heads, plan.S, D), generator=g, device="cuda") for _ in range(4))
        plan.bind_like(q)
        out, lse = torch.empty_like(q), torch.empty((1, heads, plan.S), device="cuda")
        grads = [torch.empty_like(q) for _ in range(3)]
        for name, f in (("forward", lambda: plan.forward_lse(q, k, v, out, lse)),
                        ("backward", lambda: plan.backward(do, q, k, v, out, lse, *grads))):
            f()
            best = []
            for _ in range(5):
                a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                a.record()
                for _ in range(4):
                    f()
                b.record()
                b.synchronize()
                best.append(a.elapsed_time(b))
            took[name, tile] = min(best)
        plan.destroy()
    for tile in (1, 2):
        # 280 / 68, 115 / 46 and 678 / 142 us; 92 / 199, 75 / 133 and 136 / 405 with a warp for each row
        assert took["forward", tile] <= 9 * took["forward", 32], took
        assert took["backward", tile] <= 2 * took["backward", 32], took
