"""Plans that go, or are bound anew, while a stream capture is under way: neither synchronises the device, which
would end the capture.  (A capture in the mode `global` forbids allocations everywhere and is not asked for.)"""
import threading

import pytest
import torch

from paper_2509_26538_b200 import binding as hb

pytestmark = pytest.mark.gpu


def _elsewhere(f):
    bad = []

    def go():
        try:
            f()
        except Exception as e:   # noqa: BLE001
            bad.append(e)

    t = threading.Thread(target=go)
    t.start()
    t.join()
    assert not bad, bad


@pytest.mark.parametrize("mode,here", [("thread_local", False), ("relaxed", False), ("relaxed", True)])
@pytest.mark.parametrize("what", ["destroy", "rebind"])
def test_a_capture_survives(mode, here, what):
    plan, other = hb.Plan(16, 16, 64, 5, 2, 3), hb.Plan(16, 16, 64, 0, 0, 8)
    g = torch.Generator(device="cuda")
    g.manual_seed(7)
    q, k, v = (torch.randn((1, 2, plan.S, 64), generator=g, device="cuda").bfloat16() for _ in range(3))
    out, want = torch.empty_like(q), torch.empty_like(q)
    plan.bind_like(q)
    other.bind(1, 2, 64, hb.BF16)
    plan.forward(q, k, v, want)
    torch.cuda.synchronize()
    stream, graph = torch.cuda.Stream(), torch.cuda.CUDAGraph()
    act = other.destroy if what == "destroy" else lambda: other.bind(1, 3, 64, hb.BF16)
    with torch.cuda.stream(stream):
        graph.capture_begin(capture_error_mode=mode)
        plan.forward(q, k, v, out, stream=stream)
        act() if here else _elsewhere(act)
        graph.capture_end()
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(out.view(torch.int16), want.view(torch.int16))
    hb.Plan(16, 16, 64, 1, 0, 0).destroy()   # nothing of it is left to trouble the next plan
    plan.destroy()
    other.destroy()


def test_tables_are_not_taken_from_launches_under_way():
    """A plan destroyed right behind its launches, and a new one that finds its blocks: the launches keep their tables."""
    H = W = 64
    first = hb.Plan(H, W, 512, 100, 8, 300)
    g = torch.Generator(device="cuda")
    g.manual_seed(3)
    q, k, v = (torch.randn((1, 2, first.S, 128), generator=g, device="cuda").bfloat16() for _ in range(3))
    first.bind_like(q)
    want = first.forward(q, k, v, torch.empty_like(q))
    torch.cuda.synchronize()
    stream = torch.cuda.Stream()
    for o in range(5):
        outs = [torch.empty_like(q) for _ in range(3)]
        with torch.cuda.stream(stream):
            torch.cuda._sleep(4_000_000)   # 2 ms: the launches behind it are still to come when the plan goes
            for out in outs:
                first.forward(q, k, v, out)
        first.destroy()
        second = hb.Plan(H, W, 256, 17 + o, 2, 300)
        second.bind(1, 2, 128, hb.BF16)
        torch.cuda.synchronize()
        assert all(torch.equal(want.view(torch.int16), t.view(torch.int16)) for t in outs)
        second.destroy()
        first = hb.Plan(H, W, 512, 100, 8, 300)
        first.bind_like(q)
    first.destroy()
