"""Performance cases: what users of the framework run, through its public entry points.

A program that uses the framework creates one session per network (weights on the GPU, prepacked) and keeps it.
Every batch of requests brings its own extents, so the usual call is "fresh": bind the extents, plan, launch.
Programs that meet the same extents again keep the plan ("run") or replay it as one CUDA graph ("graph"); "exact"
reads execution-determined counts back and plans the rest of the network at its true sizes.

The networks are the repository's five workloads and its two single-operator graphs.  The extents of the requests
are part of the case, the values are drawn on the GPU from the seed.  Outputs are the packed output buffers.
"""
from __future__ import annotations

import functools
import random

import torch

from paper_2403_00176_b200 import workloads as WL
from paper_2403_00176_b200.session import Session

_ESZ = {"f32": 4, "bf16": 2, "i64": 8, "bool": 1}
_DT = {"f32": torch.float32, "bf16": torch.bfloat16, "i64": torch.int64, "bool": torch.uint8}


# ------------------------------------------------------------------------------------------------ cases
def _ragged(rng, n, lo, hi):
    """Extents of n requests, each anywhere in [lo, hi]."""
    return " ".join(str(rng.randint(lo, hi)) for _ in range(n))


def _sides(rng, n):
    """n image sizes: mostly multiples of 32 as detectors resize to, one in three of any size."""
    out = []
    for _ in range(n):
        if rng.random() < 1 / 3:
            out.append("%dx%d" % (rng.randint(96, 640), rng.randint(96, 640)))
        else:
            out.append("%dx%d" % (32 * rng.randint(7, 20), 32 * rng.randint(7, 20)))
    return " ".join(out)


def _log(rng, lo, hi):
    """An integer of [lo, hi], spread over its logarithm."""
    return max(lo, min(hi, round(lo * (hi / lo) ** rng.random())))


def listed():
    r = random.Random(2403)
    return [
        # the smallest call: one fp32 fused group on one short request; launches and host work only
        {"name": "group f32, 1 request", "net": "group", "dtype": "f32", "call": "fresh", "dims": "37"},
        # an elementwise chain over activations, broadcast operand, ragged request sizes, kept plan
        {"name": "chain bf16, 4 requests", "net": "chain", "dtype": "bf16", "call": "run",
         "dims": "64x128x784 37x101x333 64x77x1024 3x250x49"},
        # execution-determined output: positions of non-zero activations, read back with their counts
        {"name": "nonzero f32, 4 requests", "net": "nonzero", "dtype": "f32", "call": "fresh",
         "dims": "1024x1024 777x1333 3x4095 2048x768"},
        # one query to a text encoder: latency of a short, odd sequence
        {"name": "encoder, 1 request", "net": "encoder", "dtype": "bf16", "call": "fresh", "dims": "127"},
        # the ordinary serving batch of the encoder: 8 sequences of 16..512 tokens
        {"name": "encoder, 8 requests", "net": "encoder", "dtype": "bf16", "call": "fresh", "dims": _ragged(r, 8, 16, 512)},
        # offline encoding of a corpus: large batches, plan kept, replayed
        {"name": "encoder, 48 requests", "net": "encoder", "dtype": "bf16", "call": "graph", "dims": _ragged(r, 48, 16, 512)},
        # one image through the token-pruning transformer, fixed resolution, replayed
        {"name": "pruning, 1 request", "net": "pruning", "dtype": "bf16", "call": "graph", "dims": "577"},
        # the ordinary batch of the token-pruning transformer: 16 images of 196..784 patches
        {"name": "pruning, 16 requests", "net": "pruning", "dtype": "bf16", "call": "fresh", "dims": _ragged(r, 16, 196, 784)},
        # one camera frame of an odd size through the convolutional stage
        {"name": "conv, 1 odd image", "net": "conv", "dtype": "bf16", "call": "fresh", "dims": "227x341"},
        # four images of different resolutions through the convolutional stage
        {"name": "conv, 4 images", "net": "conv", "dtype": "bf16", "call": "fresh", "dims": "640x480 416x416 224x608 544x320"},
        # the gated network on its ordinary batch, replayed
        {"name": "gated, 32 images", "net": "gated", "dtype": "bf16", "call": "graph", "dims": "32"},
        # the gated network where memory is short: counts read back, planned at true sizes
        {"name": "gated exact, 32 images", "net": "gated", "dtype": "bf16", "call": "exact", "dims": "32"},
    ]


def draw(rng):
    net = rng.choice(["group", "chain", "nonzero"] + ["encoder"] * 3 + ["pruning"] * 2 + ["conv"] * 2 + ["gated"] * 2)
    call = rng.choice(["fresh", "fresh", "run", "graph"])
    dtype = "bf16"
    if net == "group":
        dtype, dims = "f32", _ragged(rng, _log(rng, 1, 64), 1, 64)
    elif net == "chain":
        dtype = rng.choice(["f32", "bf16"])
        dims = " ".join("%dx%dx%d" % (_log(rng, 4, 64), _log(rng, 8, 256), _log(rng, 16, 1024)) for _ in range(_log(rng, 1, 8)))
    elif net == "nonzero":
        dtype, call = "f32", rng.choice(["fresh", "run"])
        dims = " ".join("%dx%d" % (_log(rng, 1, 2048), _log(rng, 16, 2048)) for _ in range(_log(rng, 1, 4)))
    elif net == "encoder":
        dims = _ragged(rng, _log(rng, 1, 24), 16, 512)
    elif net == "pruning":
        dims = _ragged(rng, _log(rng, 1, 20), 196, 784)
    elif net == "conv":
        dims = _sides(rng, _log(rng, 1, 4))
    else:
        call = rng.choice(["fresh", "graph", "exact"])
        dims = str(_log(rng, 1, 32))
    return {"net": net, "dtype": dtype, "call": call, "dims": dims}


# ------------------------------------------------------------------------------------------------ networks
_SYMS = {"group": ["N"], "chain": ["I", "J", "K"], "nonzero": ["R", "C"], "encoder": ["L"], "pruning": ["N0"], "conv": ["H", "W"],
         "gated": []}


def _extents(case):
    """Per request: the values of the network's symbols."""
    if case["net"] == "gated":
        return [[]]                                                # one request, the batch is a constant of the graph
    return [[int(v) for v in d.split("x")] for d in case["dims"].split()]


@functools.lru_cache(maxsize=6)
def _session(net, dtype, batch):
    """The network on the GPU, as a program keeps it between batches."""
    make = {"group": WL.cfg1, "chain": lambda: WL.fig4_chain(dtype), "nonzero": WL.nonzero_graph, "encoder": WL.cfg2, "pruning": WL.cfg3,
            "conv": WL.cfg4, "gated": lambda: WL.cfg5(B=batch)}
    return Session(make[net]())


def _kept(n0, layers):
    """Tokens that enter each layer, and those that leave the last: ceil(0.7 n) stay."""
    n = [n0]
    for _ in range(layers):
        n.append((7 * n[-1] + 9) // 10)
    return n


def _values(case, name, shape, gen):
    """One request's instance of an input, float32 on the GPU."""
    net, dev = case["net"], "cuda"
    if net == "group":
        return torch.randn(shape, generator=gen, device=dev) / 8
    if net == "nonzero":                                           # activations behind a ReLU-like sparsity of 0.6
        x = torch.randn(shape, generator=gen, device=dev)
        return x * (torch.rand(shape, generator=gen, device=dev) >= 0.6)
    if net == "pruning":
        # Patch embeddings of unit rms times the patch's salience.  Saliences come in levels, a quarter apart, as
        # many tokens in each as the network drops at that depth: which tokens are kept is then a property of the
        # input and not of the last bits of a sum, and outputs can be compared.
        _, n, d = shape
        x = torch.randn((n, d), generator=gen, device=dev)
        x = x / x.square().mean(1, keepdim=True).sqrt()
        level = torch.zeros(n, device=dev)
        for k in _kept(n, 12)[1:]:
            level[:k] += 1
        order = torch.randperm(n, generator=gen, device=dev)
        return (x * (1.25 ** level[order])[:, None])[None]
    if net == "conv":
        return torch.rand(shape, generator=gen, device=dev) * 2 - 1
    if net == "gated":                                             # per-sample contrast and per-channel offset
        b, c = shape[:2]
        gain = torch.rand((b, 1, 1, 1), generator=gen, device=dev) + 0.5
        off = torch.randn((b, c, 1, 1), generator=gen, device=dev) * 0.5
        return torch.randn(shape, generator=gen, device=dev) * gain + off
    return torch.randn(shape, generator=gen, device=dev)


class _State:
    pass


def prepare(case, seed):
    st = _State()
    st.session = s = _session(case["net"], case["dtype"], int(case["dims"]) if case["net"] == "gated" else 0)
    st.call, st.counted = case["call"], case["net"] == "nonzero"
    st.syms, st.extents = _SYMS[case["net"]], _extents(case)
    g = s.graph
    st.plan = plan = g.bind_dims(st.syms, st.extents).plan()
    gen = torch.Generator(device="cuda").manual_seed(seed)
    n = len(st.extents)

    def packed(name):
        esz = _ESZ[g.tensor_dtype(name)]
        last = plan.binding.shape(n - 1, name)
        nbytes = esz
        for d in last:
            nbytes *= d
        total = plan.instance_offset(name, n - 1) + ((nbytes + 15) & ~15)
        return torch.zeros(max(total, 16) // esz, dtype=_DT[g.tensor_dtype(name)], device="cuda")

    st.ins = []
    for name in s.in_names:
        buf = packed(name)
        for r in range(n):
            v = _values(case, name, plan.binding.shape(r, name), gen).reshape(-1)
            at = plan.instance_offset(name, r) // buf.element_size()
            buf[at:at + v.numel()] = v.to(buf.dtype)
        st.ins.append(buf)
    st.outs = [packed(name) for name in s.out_names]
    st.arena = torch.empty(max(plan.arena_bytes, 256), dtype=torch.uint8, device="cuda")
    st.in_ptrs, st.out_ptrs = [t.data_ptr() for t in st.ins], [t.data_ptr() for t in st.outs]
    if st.call == "graph":                                         # such a program captures while it sets the plan up
        plan.run_graph(st.in_ptrs, st.out_ptrs, st.arena.data_ptr(), st.arena.numel(), s.stream)
    return st


def run(st):
    s = st.session
    plan = s.graph.bind_dims(st.syms, st.extents).plan() if st.call == "fresh" else st.plan
    launch = {"graph": plan.run_graph, "exact": plan.run_exact}.get(st.call, plan.run)
    launch(st.in_ptrs, st.out_ptrs, st.arena.data_ptr(), st.arena.numel(), s.stream)
    if not st.counted:
        return dict(zip(s.out_names, st.outs))
    counts = [plan.output_shape(st.arena.data_ptr(), s.stream, r, 0)[1] for r in range(len(st.extents))]
    return {"positions": st.outs[0], "counts": counts}             # sized for the bound, zero behind what was found


# ------------------------------------------------------------------------------------------------ work and tolerance
def _transformer(counts, pairs, d, f):
    """flops of one layer over `counts` tokens whose attention has `pairs` query-key pairs"""
    return 2.0 * counts * (4 * d * d + 2 * d * f) + 4.0 * pairs * d


def work(case):
    net, esz, ext = case["net"], _ESZ[case["dtype"]], _extents(case)
    if net == "group":
        rows = 2 * sum(n for n, in ext)
        return {"bytes": 4.0 * (2 * rows * 64 + 64 * 64 + 3 * 64), "flops": 2.0 * rows * 64 * 64}
    if net == "chain":
        return {"bytes": float(esz * sum(2 * i * j * k + i for i, j, k in ext)), "flops": 0}
    if net == "nonzero":                                           # two int64 coordinates for two values in five
        return {"bytes": sum(r * c for r, c in ext) * (4 + 0.4 * 16), "flops": 0}
    if net == "encoder":
        t = sum(n for n, in ext)
        weights = 6 * (4 * 768 * 768 + 2 * 768 * 3072)
        return {"bytes": 2.0 * (2 * t * 768 + weights), "flops": 6 * _transformer(t, sum(n * n for n, in ext), 768, 3072)}
    if net == "pruning":
        flops, out = 0.0, 0.0
        for n0, in ext:
            n = _kept(n0, 12)
            flops += sum(_transformer(k, k * k, 384, 1536) for k in n[:-1])
            out += 2.0 * n[-1] * 384 + 8.0 * sum(n[1:])
        weights = 12 * (4 * 384 * 384 + 2 * 384 * 1536)
        return {"bytes": 2.0 * (sum(n for n, in ext) * 384 + weights) + out, "flops": flops}
    if net == "conv":
        px = sum(h * w for h, w in ext)
        return {"bytes": 2.0 * (2 * px * 64 + 8 * 9 * 64 * 64), "flops": 8 * 2.0 * px * 9 * 64 * 64}
    # gated: stem, projection shortcuts of every sample, half of the samples through each block's two convolutions
    b, flops, weights = int(case["dims"]), 2.0 * 112 * 112 * 64 * 147, 64 * 147
    side, cin = 112, 64
    for w in (64, 128, 256, 512):
        for k in range(4):
            down = k == 0 and w > 64
            side //= 2 if down else 1
            flops += 0.5 * 2 * side * side * 9 * w * (cin + w) + (2.0 * side * side * w * cin if down else 0)
            weights += 9 * w * (cin + w) + (w * cin if down else 0)
            cin = w
    return {"bytes": 2.0 * (b * 3 * 224 * 224 + weights + b * 512), "flops": b * flops}


def tolerance(case):
    net = case["net"]
    if net == "nonzero":
        return "exact"
    if case["dtype"] == "f32":
        return {"rel": 1e-5, "max": 1e-4}                          # sums of 64 fp32 products, one exponential
    # bf16 storage between operators: 0.0011 rms per rounding, and two correct implementations round apart
    return {"chain": {"rel": 4e-3, "max": 8e-3},                   # one rounding of the result
            "encoder": {"rel": 1.5e-2, "max": 0.2},                # about 50 roundings on the path, re-normalised
            "pruning": {"rel": 1.5e-2, "max": 0.2},                # 12 residual layers; the kept indices exactly
            "conv": {"rel": 1e-2, "max": 0.1},                     # 8 residual blocks
            "gated": {"rel": 2e-2, "max": 0.3}}[net]               # 33 convolutions; the gate bits exactly
