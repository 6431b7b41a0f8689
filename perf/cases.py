"""The work a user of this library has it do, as cases that can be timed and compared.

A case is one pass through the public binding, as a diffusion transformer calls it:

  layers  one slide cycle of a denoising step: the first layer's q, k, v are gathered into the physical
          order, every layer runs the sparse forward with its own offset, the last one writes the
          original order
  step    one attention layer with the reorder around it: three entry gathers, then the forward
          whose epilogue writes the original order
  fused   a single layer as one launch: both gathers inside the forward
  train   forward with log-sum-exp and backward on the same plan (fine-tuning through the kernel)
  host    activations in pinned host memory: copies in, one fused layer, copies out
  plan    a request at a new resolution: build the plan, bind the problem, read back the permutation
          (the caller reorders its positional encodings with it)

listed() are fixed cases, draw() gives further ones of the same ranges: token grids from 8 x 8 to
256 x 256 and short videos, nothing in them a power of two where the method allows it, 0 to 512 text
tokens, 1 to 24 heads of 64 or 128 (fp32 also 32), batches of 1 to 4, bf16 / e4m3 / fp32, the dense
[B, heads, S, D] layout and the [B, S, heads, D] layout that a projection leaves behind.
"""
from __future__ import annotations

import functools
import math
import types

import torch

from paper_2509_26538_b200 import binding as hb

_DTYPES = {"bf16": torch.bfloat16, "fp32": torch.float32, "fp8": torch.float8_e4m3fn}
_CODES = {"bf16": hb.BF16, "fp32": hb.FP32, "fp8": hb.FP8_E4M3}
_SIZE = {"bf16": 2, "fp32": 4, "fp8": 1}
# The largest amounts of arithmetic of one pass: tensor-core types, and the plain-FMA fp32 path.
_MOST_FLOPS, _MOST_FLOPS_FP32 = 4.0e12, 4.0e9


def _case(name, kind, H, W, tile, offset, shared, text, heads, dim, dtype, **more):
    c = dict(name=name, kind=kind, frames=1, H=H, W=W, tile=tile, offset=offset, shared=shared, shared_frames=0,
             text=text, batch=1, heads=heads, dim=dim, dtype=dtype, layout="bhsd", layers=1, gain=1.0)
    c.update(more)
    return c


def listed():
    return [
        # the smallest problem: four layers of a 16 x 16 grid in fp32, as a unit test or a toy model runs them
        _case("tiny_fp32_layers", "layers", 16, 16, 64, 0, 2, 0, 2, 64, "fp32", layers=4),
        # fp32 fine-tuning of a small model, or the fp32 check run beside a bf16 one
        _case("fp32_train", "train", 32, 32, 256, 128, 4, 64, 8, 64, "fp32"),
        # one layer of a thumbnail-sized latent: a call of a few microseconds
        _case("small_fused", "fused", 32, 32, 256, 128, 4, 64, 8, 128, "bf16"),
        # 1024^2 image: one slide cycle of the per-step layer schedule
        _case("img1024_layers", "layers", 64, 64, 512, 0, 8, 512, 24, 128, "bf16", layers=4),
        # 2048^2 image: one layer with the reorder around it
        _case("img2048_step", "step", 128, 128, 1024, 512, 16, 512, 24, 128, "bf16"),
        # 4096^2 image: the largest call
        _case("img4096_fwd", "layers", 256, 256, 2048, 1024, 32, 512, 24, 128, "bf16"),
        # fine-tuning at 1024^2: forward with log-sum-exp, then the backward pass
        _case("img1024_train", "train", 64, 64, 1024, 512, 8, 512, 24, 128, "bf16"),
        # 2048^2 with quantised activations
        _case("img2048_fp8_step", "step", 128, 128, 1024, 512, 16, 512, 24, 128, "fp8"),
        # a short clip of odd proportions, two prompts at once, the layout a projection leaves behind
        _case("video_d64_step", "step", 40, 72, 8192, 1000, 8, 77, 16, 64, "bf16", frames=12, shared_frames=4, batch=2,
              layout="bshd"),
        # 2048^2 with the heads of one layer cut over eight GPUs: this GPU's three
        _case("img2048_shard", "step", 128, 128, 1024, 512, 16, 512, 3, 128, "bf16"),
        # activations that live in host memory (offloaded model)
        _case("img1024_host", "host", 64, 64, 1024, 512, 8, 512, 24, 128, "bf16"),
        # a request at a new resolution
        _case("img1024_plan", "plan", 64, 64, 1024, 512, 8, 512, 24, 128, "bf16"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _padded(c):
    """(curve length, image tokens) of a case."""
    b = max(c["H"], c["W"], 1)
    b = (b - 1).bit_length()
    cells = c["frames"] * c["H"] * c["W"]
    if c["frames"] == 1:
        return 1 << (2 * b), cells
    a = max(1, (c["frames"] - 1).bit_length())
    return (1 << (3 * a) if a >= b else 1 << (2 * b + a)), cells


def _flops_estimate(c):
    np_, cells = _padded(c)
    p = c["text"] + c["shared"] ** 2 * max(1, c["shared_frames"])
    pairs = p * (c["text"] + cells) + cells * (p + max(1.0, c["tile"] * cells / np_))
    return pairs * c["batch"] * c["heads"] * c["dim"] * _flops_per_pair(c)


def draw(rng):
    kind = rng.choice(["layers", "step", "step", "fused", "train", "train", "host", "plan"])
    dtype = rng.choice(["bf16", "bf16", "bf16", "fp8", "fp32"])
    if kind == "train" and dtype == "fp8":
        dtype = "bf16"
    most = 48 if dtype == "fp32" else 64 if kind == "host" else 256
    # a grid of any proportions between 1 : 2 and 2 : 1; one in three is a square power of two
    H = _log_int(rng, 8, most)
    W = min(most, max(8, int(H * 2 ** rng.uniform(-1, 1))))
    if rng.random() < 0.33:
        H = W = 1 << (max(H, W).bit_length() - 1)
    frames = 1
    if dtype != "fp32" and kind in ("step", "fused", "train") and rng.random() < 0.25:
        frames, H, W = rng.randint(3, 16), max(8, min(H, 96) & ~1), max(8, min(W, 96) & ~1)
    c = _case("", kind, H, W, 1, 0, 0, rng.choice([0, 77, 128, 226, 333, 512, rng.randint(1, 512)]), 1, 128, dtype,
              frames=frames, layers=rng.randint(2, 4) if kind == "layers" else 1, gain=rng.choice([1.0, 1.0, 2.0]))
    del c["name"]
    c["shared"] = 2 * rng.randint(0, max(1, min(H, W) // 16))
    if frames > 1 and c["shared"]:
        c["shared_frames"] = 2 * rng.randint(1, frames // 2)
    # tiles of roughly 64 to 2048 tokens, two of them at least
    np_, cells = _padded(c)
    want = _log_int(rng, 64, 2048) * np_ / cells
    c["tile"] = 1 << max(4, min(np_.bit_length() - 2, int(round(math.log2(want)))))
    c["offset"] = rng.choice([0, c["tile"] // 2, rng.randint(0, np_ - 1)])
    c["dim"] = {"bf16": rng.choice([128, 128, 64]), "fp8": 128, "fp32": rng.choice([32, 64, 64, 128])}[dtype]
    c["heads"], c["batch"] = rng.choice([1, 2, 3, 5, 8, 12, 16, 24]), rng.choice([1, 1, 2, 4])
    if kind != "host":
        c["layout"] = rng.choice(["bhsd", "bshd"])
    limit = (_MOST_FLOPS_FP32 if dtype == "fp32" else _MOST_FLOPS) * (0.02 if kind == "host" else 1.0)
    while _flops_estimate(c) > limit and c["batch"] * c["heads"] > 1:
        if c["batch"] > 1:
            c["batch"] -= 1
        else:
            c["heads"] -= 1
    return c


def _new_plan(c, layer=0):
    offset = c["offset"] + layer * c["tile"] // 4
    if c["frames"] > 1:
        return hb.Plan(c["H"], c["W"], c["tile"], offset, c["shared"], c["text"], frames=c["frames"],
                       shared_frames=c["shared_frames"])
    return hb.Plan(c["H"], c["W"], c["tile"], offset, c["shared"], c["text"])


def _empty(c, S, dtype):
    """A [B, heads, S, D] view in the case's layout."""
    if c["layout"] == "bhsd":
        return torch.empty((c["batch"], c["heads"], S, c["dim"]), dtype=dtype, device="cuda")
    return torch.empty((c["batch"], S, c["heads"], c["dim"]), dtype=dtype, device="cuda").transpose(1, 2)


def _rows(c, t):
    """The same memory as the [..., S, row] array the gathers take."""
    return t if c["layout"] == "bhsd" else t.transpose(1, 2).flatten(2)


def _normal(c, S, g, gain=1.0):
    t = _empty(c, S, _DTYPES[c["dtype"]])
    # values: normalised queries and keys, N(0, 1); `gain` sharpens the softmax as a learned norm weight does
    t.copy_(torch.randn(t.shape, generator=g, device="cuda") * gain)
    return t


def prepare(case, seed):
    c = dict(case)
    st = types.SimpleNamespace(case=c)
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    if c["kind"] == "plan":
        # another request: the offset is what changes from layer to layer and from seed to seed
        c["offset"] += 1 + seed % 997
        return st
    st.plans = [_new_plan(c, layer) for layer in range(c["layers"])]
    S = st.plans[0].S
    st.qkv = [[_normal(c, S, g, c["gain"]), _normal(c, S, g), _normal(c, S, g)] for _ in range(c["layers"])]
    out_dtype = torch.bfloat16 if c["dtype"] == "fp8" else _DTYPES[c["dtype"]]
    st.out = [_empty(c, S, out_dtype) for _ in range(c["layers"])]
    for p in st.plans:
        p.bind_like(st.qkv[0][0])
    if c["kind"] in ("layers", "step"):
        st.first = [_empty(c, S, _DTYPES[c["dtype"]]) for _ in range(3)]
    elif c["kind"] == "train":
        st.lse = torch.empty((c["batch"], c["heads"], S), dtype=torch.float32, device="cuda")
        st.dout = _normal(c, S, g)
        st.grads = [_empty(c, S, out_dtype) for _ in range(3)]
    elif c["kind"] == "host":
        st.qkv = [[t.cpu().pin_memory() for t in st.qkv[0]]]
        st.out = [torch.empty(st.out[0].shape, dtype=out_dtype).pin_memory()]
    return st


def run(st):
    c = st.case
    kind = c["kind"]
    if kind == "plan":
        plan = _new_plan(c)
        plan.bind(c["batch"], c["heads"], c["dim"], _CODES[c["dtype"]])
        got = [plan.export(hb.EXPORT_PHYS2ORIG), plan.export(hb.EXPORT_WINDOWS)]
        plan.destroy()
        return got
    if kind in ("layers", "step"):
        last = len(st.plans) - 1
        for src, dst in zip(st.qkv[0], st.first):
            st.plans[0].permute(_rows(c, src), _rows(c, dst))
        for layer, plan in enumerate(st.plans):
            q, k, v = st.first if layer == 0 else st.qkv[layer]
            if layer < last:
                plan.forward(q, k, v, st.out[layer])
            else:
                plan.forward_unpermute(q, k, v, st.out[layer])
        return st.out
    (q, k, v), plan, out = st.qkv[0], st.plans[0], st.out[0]
    if kind == "fused":
        return plan.forward_fused(q, k, v, out)
    if kind == "host":
        return plan.forward_host(q, k, v, out)
    plan.forward_lse(q, k, v, out, st.lse)
    plan.backward(st.dout, q, k, v, out, st.lse, *st.grads)
    return [out, st.lse] + st.grads


def _flops_per_pair(c):
    """Per kept (query, key) pair and unit of head dim: two contractions forward, five backward."""
    return {"plan": 0, "train": 14}.get(c["kind"], 4 * c["layers"])


@functools.lru_cache(maxsize=None)
def _pairs(frames, H, W, tile, offset, shared, shared_frames, text):
    plan = hb.Plan(H, W, tile, offset, shared, text, frames=frames, shared_frames=shared_frames)
    return int(plan.export(hb.EXPORT_NNZ)[0]), int(plan.export(hb.EXPORT_INFO)[7]), plan.S


def work(case):
    c = case
    pairs, tiles, S = _pairs(c["frames"], c["H"], c["W"], c["tile"], c["offset"], c["shared"], c["shared_frames"], c["text"])
    if c["kind"] == "plan":
        return {"bytes": 4 * S + 20 * tiles, "flops": 0}   # the permutation and the tile table, written once
    elems = c["batch"] * c["heads"] * S * c["dim"]
    e_in, e_out = _SIZE[c["dtype"]], 2 if c["dtype"] == "fp8" else _SIZE[c["dtype"]]
    moved = c["layers"] * elems * (3 * e_in + e_out)
    if c["kind"] == "train":
        moved = elems * 8 * e_in + 4 * c["batch"] * c["heads"] * S   # q k v dout in; out dq dk dv and the log-sum-exp out
    return {"bytes": moved, "flops": pairs * c["batch"] * c["heads"] * c["dim"] * _flops_per_pair(c)}


def tolerance(case):
    """About four times the distance of the path from itself in 64 bits, measured on the small cases."""
    if case["kind"] == "plan":
        return "exact"
    if case["dtype"] == "fp32":
        return {"rel": 3e-6}    # sums of up to a few thousand 32-bit products: 2.5e-7 ... 7e-7
    if case["dtype"] == "fp8":
        return {"rel": 8e-2}    # weights rounded to 3 mantissa bits: 1.6e-2 ... 2.5e-2
    return {"rel": 1e-2}        # weights and results rounded to 8 bits: 1.9e-3 ... 2.8e-3
