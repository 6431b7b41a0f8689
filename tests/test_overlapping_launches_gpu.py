"""Launches overlap the drain of the one before them: a chain of calls that reuse each other's buffers gives,
bit for bit, what the same calls give one at a time."""
import pytest
import torch

from paper_2509_26538_b200 import binding as hb

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,W,tile,o,hs,nt,B,heads,D,dtype", [
    (8, 8, 16, 3, 2, 5, 1, 2, 64, torch.float32),
    (16, 16, 64, 9, 2, 0, 1, 2, 128, torch.bfloat16),      # few CTAs: the next kernel starts on idle SMs
    (32, 32, 256, 128, 4, 64, 1, 8, 128, torch.bfloat16),  # clusters
    (40, 24, 256, 77, 4, 33, 2, 5, 64, torch.bfloat16),
    (64, 64, 512, 100, 8, 300, 1, 24, 128, torch.bfloat16),
])
def test_chain_equals_single_steps(H, W, tile, o, hs, nt, B, heads, D, dtype):
    plan = hb.Plan(H, W, tile, o, hs, nt)
    g = torch.Generator(device="cuda")
    g.manual_seed(H + D)
    x = [torch.randn((B, heads, plan.S, D), generator=g, device="cuda").to(dtype) for _ in range(4)]
    plan.bind_like(x[0])

    def chain(step):
        q, k, v, do = (t.clone() for t in x)
        p = [torch.empty_like(q) for _ in range(4)]
        out, grads = torch.empty_like(q), [torch.empty_like(q) for _ in range(3)]
        lse = torch.empty((B, heads, plan.S), device="cuda")
        torch.cuda.synchronize()
        for _ in range(6):
            for src, dst in zip((q, k, v, do), p):
                step(plan.permute, src, dst)
            step(plan.forward_lse, p[0], p[1], p[2], out, lse)
            step(plan.backward, p[3], p[0], p[1], p[2], out, lse, *grads)
            step(plan.unpermute, out, q)             # the next round's query: read by the first kernel above
            step(plan.forward, p[1], p[0], p[2], out)   # and the output written again right behind its reader
            step(plan.forward_fused, q, k, v, do)
        torch.cuda.synchronize()
        assert plan.status() == 0
        return [q, do, out, lse] + grads

    def one_at_a_time(f, *args):
        f(*args)
        torch.cuda.synchronize()

    for a, b in zip(chain(lambda f, *args: f(*args)), chain(one_at_a_time)):
        assert torch.equal(a.view(torch.uint8), b.view(torch.uint8))
    plan.destroy()


@pytest.mark.parametrize("tile,nt,heads", [(256, 64, 48), (512, 512, 48), (1024, 512, 24)])
def test_launches_in_a_row_take_no_longer_than_apart(tile, nt, heads):
    """Launches that fill the chip, right behind each other and with another kernel of a few microseconds between any
    two: overlapping ones took 15 to 27 % longer in a row."""
    plan = hb.Plan(64, 64, tile, tile // 2, 4 if nt == 64 else 8, nt)
    g = torch.Generator(device="cuda")
    g.manual_seed(1)
    x = [torch.randn((1, heads, plan.S, 128), generator=g, device="cuda").bfloat16() for _ in range(3)]
    plan.bind_like(x[0])
    if plan.export(hb.EXPORT_CUTS)[0, 0] != 1:
        pytest.skip("cut on this device, where overlapping pays")
    out, small = torch.empty_like(x[0]), torch.zeros(1024, device="cuda")

    def took(apart):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        for _ in range(8):
            plan.forward_fused(*x, out)
            if apart:
                small.add_(1)
        b.record()
        b.synchronize()
        return a.elapsed_time(b)

    took(False), took(True)
    pairs = [(took(False), took(True)) for _ in range(15)]
    in_a_row, apart = (sorted(p[i] for p in pairs)[7] for i in (0, 1))
    assert in_a_row <= 1.08 * apart, (in_a_row / 8, apart / 8)
    plan.destroy()
