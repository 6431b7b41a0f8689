"""hilberta_forward_host at sizes from one slice of heads to eight (a launch each), prime numbers of heads and batches among
them, equals the fused launch on device buffers bit for bit (a slice's rows are summed in the same order)."""
import pytest
import torch

from paper_2509_26538_b200 import binding as hb

pytestmark = pytest.mark.gpu


def _check(plan, batch, heads, dim, dtype, slices):
    kind = torch.float8_e4m3fn if dtype == "fp8" else torch.bfloat16
    g = torch.Generator(device="cuda").manual_seed(plan.S + heads)
    q, k, v = (torch.randn((batch, heads, plan.S, dim), generator=g, device="cuda").to(kind) for _ in range(3))
    plan.bind_like(q)
    want = torch.empty(q.shape, dtype=torch.bfloat16, device="cuda")
    plan.forward_fused(q, k, v, want)
    hq, hk, hv = (t.cpu().pin_memory() for t in (q, k, v))
    out = torch.empty(q.shape, dtype=torch.bfloat16).pin_memory()
    for _ in range(2):
        out.fill_(7.0)
        before = hb.launch_count()
        plan.forward_host(hq, hk, hv, out)
        assert hb.launch_count() - before == slices
        assert torch.equal(out, want.cpu())
    assert plan.status() == 0


@pytest.mark.parametrize("H,text,batch,heads,dim,dtype,slices", [
    (8, 0, 1, 1, 64, "bf16", 1), (16, 5, 1, 7, 128, "bf16", 1), (16, 0, 3, 6, 64, "bf16", 1),
    (40, 77, 1, 13, 128, "bf16", 2),                                                   # 7 and 6 heads
    (64, 512, 1, 24, 128, "bf16", 4), (64, 512, 1, 24, 128, "fp8", 4), (48, 33, 4, 10, 128, "bf16", 5),
    (64, 333, 2, 7, 128, "fp8", 4), (88, 256, 1, 31, 128, "bf16", 6), (64, 512, 1, 67, 64, "bf16", 5),
    (96, 512, 2, 16, 128, "bf16", 8), (128, 512, 1, 23, 128, "bf16", 7), (96, 512, 1, 10, 128, "bf16", 5),
    (96, 512, 2, 20, 64, "bf16", 8), (56, 333, 1, 24, 64, "bf16", 3),
])
def test_host_slices(H, text, batch, heads, dim, dtype, slices):
    plan = hb.Plan(H, H, 64, 16, 2, text)
    _check(plan, batch, heads, dim, dtype, slices)
    plan.destroy()


@pytest.mark.parametrize("H,tile,shared,text,batch,heads,dim,dtype,slices", [
    (128, 1024, 16, 512, 1, 3, 128, "bf16", 3), (128, 1024, 16, 512, 1, 3, 128, "fp8", 3),
    (128, 1024, 16, 512, 1, 5, 64, "bf16", 2),                                         # 3 and 2 heads
    (64, 512, 8, 512, 2, 3, 64, "bf16", 2), (64, 512, 8, 512, 3, 2, 128, "bf16", 2),
])
def test_host_slices_of_cut_lists(H, tile, shared, text, batch, heads, dim, dtype, slices):
    """Key lists cut over clusters: the shares are those of the whole problem, the schedules the slices' own."""
    plan = hb.Plan(H, H, tile, 0, shared, text)
    _check(plan, batch, heads, dim, dtype, slices)
    cluster, items, _ = plan.export(hb.EXPORT_CUTS)[0]
    assert cluster > 1 and items > 0
    plan.destroy()


@pytest.mark.parametrize("pinned", [(True, False), (False, True), (False, False)])
def test_pageable_buffers(pinned):
    """A copy to pageable memory ends before the next one begins: one slice, while pageable inputs keep theirs."""
    plan = hb.Plan(64, 64, 64, 16, 2, 512)
    g = torch.Generator(device="cuda").manual_seed(3)
    q, k, v = (torch.randn((1, 24, plan.S, 128), generator=g, device="cuda").bfloat16() for _ in range(3))
    plan.bind_like(q)
    want = plan.forward_fused(q, k, v, torch.empty_like(q)).cpu()
    ins = [t.cpu().pin_memory() if pinned[0] else t.cpu() for t in (q, k, v)]
    out = torch.full(q.shape, 7.0, dtype=torch.bfloat16)
    out = out.pin_memory() if pinned[1] else out
    before = hb.launch_count()
    plan.forward_host(*ins, out)
    launches = hb.launch_count() - before
    assert torch.equal(out, want)
    assert launches == 1 if not pinned[1] else launches > 1
    plan.destroy()


def test_slices_after_another_bind():
    """The slices' schedules belong to the binding: other heads, types and cuts in between, in the same workspace, on
    other streams and with a pageable output."""
    plan = hb.Plan(64, 64, 512, 0, 8, 512)
    shapes = [(1, 13, 128, "bf16", 3), (2, 3, 64, "bf16", 2), (1, 24, 128, "fp8", 4), (1, 5, 128, "bf16", 2)]
    for shape in shapes + shapes[::-1]:
        with torch.cuda.stream(torch.cuda.Stream()):
            _check(plan, *shape)
    plan.destroy()
    # the first call on a binding in one slice, the next in two, again in one
    plan = hb.Plan(64, 64, 512, 0, 8, 512)
    q, k, v = (torch.randn((1, 5, plan.S, 128), device="cuda").bfloat16() for _ in range(3))
    plan.bind_like(q)
    want = plan.forward_fused(q, k, v, torch.empty_like(q)).cpu()
    pageable = [t.cpu() for t in (q, k, v, torch.zeros_like(q))]
    pinned = [t.pin_memory() for t in pageable]
    for buffers, slices in ((pageable, 1), (pinned, 2), (pageable, 1), (pinned, 2)):
        buffers[3].fill_(7.0)
        before = hb.launch_count()
        plan.forward_host(*buffers)
        assert hb.launch_count() - before == slices
        assert torch.equal(buffers[3], want)
    assert plan.status() == 0
    plan.destroy()
