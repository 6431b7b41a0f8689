"""What cut lists can meet: several cut units in a CTA one after the other (of two query tiles, then of one), clusters
of every size in both directions, the layout a projection leaves behind, sharp softmax rows, video volumes and
equal groups.  Each case states the cuts that it is there for, so that it cannot come to test nothing.
Against the definition in 64 bits on the GPU, twice bit for bit."""
import math

import numpy as np
import pytest
import torch

from paper_2509_26538_b200 import binding as hb

pytestmark = pytest.mark.gpu


def _groups(plan, P):
    """Physical row -> tile, -1 for the prefix."""
    group = torch.full((plan.S,), -1, dtype=torch.int64)
    for t, (_, a, n, b, m) in enumerate(plan.export(hb.EXPORT_WINDOWS).tolist()):
        group[a:a + n] = t
        group[b:b + m] = t
    assert (group[P:] >= 0).all() and (group[:P] == -1).all()
    return group.cuda()


def _exact(q, k, v, do, keep):
    """out, log-sum-exp, dq, dk, dv of one head in 64 bits."""
    q, k, v, do = (t.double() for t in (q, k, v, do))
    s = (q @ k.T / math.sqrt(q.shape[1])).masked_fill_(~keep, -math.inf)
    lse = torch.logsumexp(s, 1)
    p = s.sub_(lse[:, None]).exp_()
    out = p @ v
    dv = p.T @ do
    ds = (do @ v.T - (do * out).sum(1, keepdim=True)).mul_(p).div_(math.sqrt(q.shape[1]))
    return out, lse, ds @ k, ds.T @ q, dv


CASES = {
    # name: (plan arguments, plan options, batch, heads, head dim, type, layout, gain of q, forward cuts, backward cuts)
    # cuts: at least so many cut units in a CTA (how large the clusters are depends on how many of each size the
    # device runs at once; here 2, 4 and 8 all come up, see the last test)
    "dense_nine_heads": ((64, 64, 4096, 0, 0, 1), {}, 1, 9, 128, "bf16", "bhsd", 1, 3, None),
    "dense_nine_heads_fp8": ((64, 64, 4096, 0, 0, 1), {}, 1, 9, 128, "fp8", "bhsd", 1, 3, None),
    "dense_large": ((96, 96, 16384, 0, 0, 333), {}, 1, 2, 64, "bf16", "bhsd", 1, 3, 3),
    "dense_large_strided": ((96, 96, 16384, 0, 0, 333), {}, 2, 1, 128, "bf16", "bshd", 2, 3, 3),
    "prefix_strided": ((48, 40, 1024, 77, 8, 226), {}, 1, 2, 64, "bf16", "bshd", 1, 1, 1),
    "prefix_two_batches": ((64, 64, 512, 0, 8, 512), {}, 3, 1, 64, "bf16", "bshd", 4, 1, 1),
    "prefix_many_heads": ((48, 64, 512, 3257, 4, 64), {}, 1, 12, 128, "bf16", "bhsd", 1, 1, 1),
    "prefix_fp8_strided": ((48, 40, 1024, 77, 8, 226), {}, 1, 2, 128, "fp8", "bshd", 2, 1, None),
    "video": ((12, 20, 1024, 999, 2, 300), dict(frames=5, shared_frames=2), 1, 4, 128, "bf16", "bhsd", 2, 1, 1),
    "groups": ((48, 48, 0, 100, 8, 300), dict(groups=5), 1, 2, 128, "bf16", "bshd", 1, 1, 1),
}


@pytest.mark.parametrize("name", CASES)
def test_against_the_definition(name):
    args, more, B, heads, D, kind, layout, gain, forward, backward = CASES[name]
    plan = hb.Plan(*args, **more)
    S = plan.S
    dt = torch.float8_e4m3fn if kind == "fp8" else torch.bfloat16
    g = torch.Generator(device="cuda")
    g.manual_seed(S + D)

    def tensor(dtype):
        if layout == "bhsd":
            return torch.full((B, heads, S, D), float("nan"), dtype=dtype, device="cuda")
        return torch.full((B, S, heads, D), float("nan"), dtype=dtype, device="cuda").transpose(1, 2)

    def normal(scale=1.0):
        t = tensor(dt)
        t.copy_(torch.randn(t.shape, generator=g, device="cuda") * scale)
        return t

    q, k, v, do = normal(gain), normal(), normal(), normal()
    plan.bind_like(q)
    cuts = plan.export(hb.EXPORT_CUTS).tolist()
    assert cuts[0][0] > 1 and cuts[0][1] > 0 and cuts[0][2] >= forward, cuts
    if backward:
        assert cuts[1][0] > 1 and cuts[1][1] > 0 and cuts[1][2] >= backward, cuts
    info = plan.export(hb.EXPORT_INFO)
    group = _groups(plan, int(info[5] + info[6]))
    keep = (group[:, None] == -1) | (group[None, :] == -1) | (group[:, None] == group[None, :])

    runs = []
    for _ in range(2):
        out, lse = tensor(torch.bfloat16), torch.full((B, heads, S), float("nan"), device="cuda")
        plan.forward_lse(q, k, v, out, lse)
        grads = [tensor(torch.bfloat16) for _ in range(3)] if backward else []
        if backward:
            plan.backward(do, q, k, v, out, lse, *grads)
        runs.append([out, lse] + grads)
    # the same rows by the other ways through: original order in and out
    order = torch.from_numpy(plan.export(hb.EXPORT_PHYS2ORIG).astype(np.int64)).cuda()
    back = torch.empty_like(order)
    back[order] = torch.arange(S, device="cuda")
    fused, unpermuted = tensor(torch.bfloat16), tensor(torch.bfloat16)
    x = [tensor(dt) for _ in range(3)]
    byte = torch.uint8 if kind == "fp8" else torch.int16
    for src, dst in zip((q, k, v), x):
        dst.view(byte).copy_(src.view(byte)[:, :, back])
    plan.forward_fused(*x, fused)
    plan.forward_unpermute(q, k, v, unpermuted)
    assert plan.status() == 0
    for a, b in zip(*runs):
        assert torch.equal(a.contiguous().view(torch.uint8), b.contiguous().view(torch.uint8))
    want = runs[0][0][:, :, back].contiguous().view(torch.int16)
    assert torch.equal(fused.contiguous().view(torch.int16), want)
    assert torch.equal(unpermuted.contiguous().view(torch.int16), want)

    # the bars of the uncut kernels
    vmax = float(v.float().abs().max())
    bar = (2 ** -4 * vmax + 1e-2, 4e-2) if kind == "fp8" else (1e-2 * max(1.0, vmax / 4), 5e-3)
    for b in range(B):
        for h in range(heads):
            ref = _exact(q[b, h], k[b, h], v[b, h], do[b, h], keep)
            got = [t[b, h].double() for t in runs[0]]
            assert (got[0] - ref[0]).abs().max() <= bar[0] and (got[0] - ref[0]).norm() <= bar[1] * ref[0].norm()
            assert (got[1] - ref[1]).abs().max() <= 2e-3
            for mine, r in zip(got[2:], ref[2:]):
                assert (mine - r).norm() <= 5e-3 * r.norm()
                assert (mine - r).abs().max() <= 1e-2 * max(1.0, float(r.abs().max()))
    plan.destroy()


@pytest.mark.parametrize("shape,forward,backward", [
    # of tests/test_attn_split_gpu.py and tests/test_backward_split_gpu.py
    ((16, 32, 256, 100, 2, 20, 1, 1), False, False),
    ((32, 32, 256, 128, 4, 64, 1, 8), True, None),
    ((48, 40, 1024, 77, 8, 226, 1, 2), True, True),
    ((48, 40, 1024, 77, 8, 226, 3, 5), True, None),
    ((64, 64, 512, 0, 8, 512, 1, 3), True, True),
    ((64, 64, 4096, 0, 0, 1, 1, 1), True, True),
    ((48, 48, 4096, 0, 0, 1, 1, 1), True, True),
])
def test_which_shapes_are_cut(shape, forward, backward):
    plan = hb.Plan(*shape[:6])
    with pytest.raises(hb.HilbertaError):
        plan.export(hb.EXPORT_CUTS)   # of the binding
    plan.bind(shape[6], shape[7], 128, hb.BF16)
    cuts = plan.export(hb.EXPORT_CUTS)
    for want, (cluster, items, most) in zip((forward, backward), cuts.tolist()):
        assert want is None or (cluster > 1) == want
        assert (cluster > 1) == (items > 0) == (most > 0)
    plan.destroy()


def test_clusters_of_every_size_come_up():
    seen = [set(), set()]   # forward, backward
    for args, more, B, heads, D, kind, *_ in CASES.values():
        plan = hb.Plan(*args, **more)
        plan.bind(B, heads, D, hb.FP8_E4M3 if kind == "fp8" else hb.BF16)
        for s, c in zip(seen, plan.export(hb.EXPORT_CUTS)[:, 0].tolist()):
            s.add(c)
        plan.destroy()
    assert {2, 4, 8} <= seen[0] | seen[1] and min(len(s - {1}) for s in seen) >= 2, seen
