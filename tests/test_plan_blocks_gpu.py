"""Plans that come and go: tables built in a block that another plan or binding has left behind are the
plan's own, rebinding included, from several threads at once."""
import threading

import numpy as np
import pytest
import torch

from oracle import hilberta_oracle as orc
from paper_2509_26538_b200 import binding as hb

pytestmark = pytest.mark.gpu

SHAPES = [(16, 16, 64, 5, 2, 7), (32, 24, 256, 100, 4, 0), (8, 8, 16, 3, 0, 33), (48, 48, 512, 7, 8, 300)]


def test_blocks_are_reused_from_several_threads():
    ref = {s: orc.plan_arrays(*s) for s in SHAPES}
    bad = []

    def work(k):
        torch.cuda.set_device(0)
        stream = torch.cuda.Stream()
        for i in range(12):
            s = SHAPES[(i + k) % len(SHAPES)]
            plan = hb.Plan(*s)
            S = plan.S
            g = torch.Generator(device="cuda")
            g.manual_seed(i)
            with torch.cuda.stream(stream):
                q, kk, v = (torch.randn((1, 2, S, 64), generator=g, device="cuda") for _ in range(3))
                b = [t.to(torch.bfloat16) for t in (q, kk, v)]
                plan.bind_like(b[0])
                one = plan.forward(*b, torch.empty_like(b[0]))
                plan.bind_like(q)              # another binding takes the first one's place
                two = plan.forward(q, kk, v, torch.empty_like(q))
                stream.synchronize()
                # bf16 operands and weights: 2^-9 each, N(0, 1) values
                if not (torch.isfinite(two).all() and (one.float() - two).norm() <= 1e-2 * two.norm()):
                    bad.append((k, i, "forward"))
            for what, key in ((hb.EXPORT_PHYS2ORIG, "phys2orig"), (hb.EXPORT_WINDOWS, "windows")):
                if not np.array_equal(plan.export(what), ref[s][key]):
                    bad.append((k, i, key))
            plan.destroy()

    threads = [threading.Thread(target=work, args=(k,)) for k in range(3)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad, bad


def test_kept_memory_is_bounded_recent_and_given_back():
    hb.trim()
    assert hb.trim() == 0
    small = [hb.Plan(16, 16, 64, o, 2, 7) for o in range(40)]
    for p in small:
        p.destroy()
    held = hb.trim()
    assert 0 < held <= 16 * 65536 * 2
    # many small blocks do not keep a larger one out
    small = [hb.Plan(16, 16, 64, o, 2, 7) for o in range(40)]
    for p in small:
        p.destroy()
    large = hb.Plan(64, 64, 256, 0, 0, 0)
    large.bind(1, 64, 64, hb.FP32)          # two floats per row: 2 MB
    large.destroy()
    assert hb.trim() >= 64 * 4096 * 2 * 4
    # nor do many large ones add up
    plans = [hb.Plan(128, 128, 1024, o, 0, 0) for o in range(8)]
    for p in plans:
        p.bind(2, 48, 64, hb.FP32)          # 12 MB each
    for p in plans:
        p.destroy()
    assert 48 << 20 <= hb.trim() <= 64 << 20


def test_the_workspace_of_host_calls_is_kept_too():
    """The first host-buffer call on a plan finds the workspace that an earlier plan's calls have left."""
    hb.trim()
    host = [torch.randn((1, 2, 64 * 64, 128)).bfloat16().pin_memory() for _ in range(4)]
    want = None
    for i in range(3):
        plan = hb.Plan(64, 64, 256, 9, 4, 0)
        plan.bind(1, 2, 128, hb.BF16)
        before = torch.cuda.mem_get_info()[0]
        plan.forward_host(*host)
        if i:
            assert torch.cuda.mem_get_info()[0] == before
            assert torch.equal(host[3].view(torch.int16), want.view(torch.int16))
        want = host[3].clone()
        plan.destroy()
    assert hb.trim() >= 4 * host[0].nbytes


@pytest.mark.skipif(torch.cuda.device_count() < 2, reason="two devices")
def test_a_plan_is_bound_on_its_own_device():
    """Whichever device is current: tables, kernel attributes and results are those of the plan's device, which a
    bind elsewhere must not have marked as set up."""
    with torch.cuda.device(1):
        plan = hb.Plan(24, 24, 64, 5, 2, 40)
        x = [torch.randn((1, 2, plan.S, 128), device="cuda") for _ in range(3)]
    plan.bind_like(x[0])   # device 0 is current; fp32 of head dim 128 needs the opt-in to large shared memory
    assert torch.cuda.current_device() == 0
    with torch.cuda.device(1):
        out = plan.forward(*x, torch.full_like(x[0], float("nan")))
        assert torch.isfinite(out).all() and plan.status() == 0
    plan.destroy()
