"""The timed cases: what a training program has the library do, through the binding's public calls.

A program that checkpoints with it keeps a tracked state on the GPU, compresses every snapshot against it (advancing
the tracked state in the same call, or only for the stream), and after a failure recovers a state from a base and the
streams that lead from it, one after the other or the whole vector at once. Sizes are the four model states of
``synth.CONFIGS`` (61,706 to 1,315,575,808 fp32 values) and a single small layer; ``draw`` spreads over the same
range. All buffers that such a program keeps (streams, workspace, outputs) are made once in ``prepare``. Streams and
recovered states are exact: streams byte for byte, states bit for bit.
"""
from __future__ import annotations

import dataclasses
import math
import random

import torch

from paper_2009_13003_b200 import binding, synth

DEVICE = "cuda:0"


def listed():
    return [
        # one bias or normalisation layer of a model that is checkpointed tensor by tensor: nothing but latency
        {"name": "layer snapshot", "op": "snapshot", "state": "gauss", "n": 1000, "nbits": 4},
        # a small model's snapshot, stored at once (so its size is needed), and the state recovered from it
        {"name": "lenet5 compress", "op": "compress", "state": "lenet5", "n": 61_706, "nbits": 3},
        {"name": "lenet5 recover", "op": "recover", "state": "lenet5", "n": 61_706, "nbits": 3, "k": 1},
        # a mid-sized model: the snapshot inside the training loop, and the restart from a base and ten snapshots
        {"name": "resnet18 snapshot", "op": "snapshot", "state": "resnet18", "n": 11_689_512, "nbits": 4},
        {"name": "resnet18 recover 10", "op": "recover", "state": "resnet18", "n": 11_689_512, "nbits": 4, "k": 10},
        # the same model layer by layer: 62 tensors of 64 to 2.4 million values, a stream for each
        {"name": "resnet18 layers snapshot", "op": "layers_snapshot", "state": "resnet18", "n": 11_689_512, "nbits": 4, "layers": 62},
        {"name": "resnet18 layers recover", "op": "layers_recover", "state": "resnet18", "n": 11_689_512, "nbits": 4, "layers": 62, "k": 1},
        # a large model with frozen parts
        {"name": "vgg16 compress", "op": "compress", "state": "vgg16", "n": 138_357_544, "nbits": 4},
        {"name": "vgg16 recover", "op": "recover", "state": "vgg16", "n": 138_357_544, "nbits": 4, "k": 1},
        # checkpoint merging: a chain replaced by one stream, when old snapshots are pruned; a ragged size
        {"name": "merge 4", "op": "merge", "state": "lognormal", "n": 20_000_003, "nbits": 6, "k": 4},
        # the largest state, both directions
        {"name": "xfmr1p3b compress", "op": "compress", "state": "xfmr1p3b", "n": 1_315_575_808, "nbits": 5},
        {"name": "xfmr1p3b recover 4", "op": "recover", "state": "xfmr1p3b", "n": 1_315_575_808, "nbits": 5, "k": 4},
    ]


def draw(rng):
    op = rng.choice(["snapshot", "compress", "compress", "recover", "recover", "layers_snapshot", "layers_recover", "merge"])
    state = rng.choice(["gauss", "laplace", "lognormal", "student"])
    hi = {"layers_snapshot": 24.0, "layers_recover": 24.0, "merge": 27.0}.get(op, 28.0)
    case = {"op": op, "state": state, "n": int(2.0 ** rng.uniform(8.0, hi)), "nbits": rng.choice([2, 3, 4, 4, 5, 6, 8])}
    if op.startswith("layers"):
        case["n"] = max(4096, case["n"] // 4 * 4)  # layers start at multiples of four values
        case["layers"] = rng.randint(4, 48)
    if op == "recover":
        case["k"] = rng.choice([1, 1, 2, 3, 4, 6, 8])
    if op == "layers_recover":
        case["k"] = rng.choice([1, 2, 4])
    if op == "merge":
        case["k"] = rng.randint(2, 8)
    return case


def _segments(case):
    """Layer boundaries: of the ResNet-18-sized state its own tensors, else large and small layers in turn."""
    if case["state"] == "resnet18":
        sizes = synth.resnet18_segments()
    else:
        rng = random.Random(case["n"] * 64 + case["layers"])
        share = [2.0 ** rng.uniform(-8.0, 0.0) for _ in range(case["layers"])]
        sizes = [max(4, int(case["n"] * s / sum(share)) // 4 * 4) for s in share]
        sizes[-1] += case["n"] - sum(sizes)
        if sizes[-1] < 0:
            raise ValueError("too many layers for this size")
    begin = [0]
    for s in sizes:
        begin.append(begin[-1] + s)
    return begin


def _base(case, seed):
    if case["state"] in synth.CONFIGS:
        cfg = dataclasses.replace(synth.CONFIGS[case["state"]], seed=seed * 100_003)
        return synth.base_state(cfg, DEVICE, case["n"])
    return synth.normal(case["n"], 0.02, DEVICE, seed * 100_003)


def _delta(case, seed, t):
    """The t-th update of the state (1-based)."""
    n, state = case["n"], case["state"]
    if state in synth.CONFIGS:
        return synth.snapshot_delta(dataclasses.replace(synth.CONFIGS[state], seed=seed * 100_003), t, DEVICE, n)
    if state == "student":
        return synth.student_t3(n, 1e-4, DEVICE, seed * 100_003 + t)
    return synth.sweep_delta(state, n, DEVICE, seed * 100_003 + t)


def prepare(case, seed):
    op, n, nbits = case["op"], case["n"], case["nbits"]
    base = _base(case, seed)
    s = {"op": op, "base": base, "nbits": nbits}
    if op.startswith("layers"):
        s["seg"] = seg = _segments(case)
        longest = max(b - a for a, b in zip(seg[:-1], seg[1:]))
        total = binding.segments_layout(seg, nbits)[1]
    if op in ("compress", "snapshot", "layers_snapshot"):
        s["cur"] = base + _delta(case, seed, 1)
        # zeroed, so that the bytes behind a stream's end compare equal
        s["stream"] = torch.zeros(total if op == "layers_snapshot" else binding.stream_bound(n, nbits), dtype=torch.uint8, device=DEVICE)
        s["workspace"] = binding.alloc_workspace(longest if op == "layers_snapshot" else n, DEVICE)
        if op != "compress":
            s["tracked"] = torch.empty_like(base)
        return s
    # the streams of a run of snapshots, each against the state that the streams before it recover
    tracked, cur, streams = base.clone(), base.clone(), []
    workspace = binding.alloc_workspace(n, DEVICE)
    buffer = torch.empty(total if op == "layers_recover" else binding.stream_bound(n, nbits), dtype=torch.uint8, device=DEVICE)
    for t in range(1, case["k"] + 1):
        cur += _delta(case, seed, t)
        if op == "layers_recover":
            binding.compress_segments(tracked, cur, seg, nbits, buffer, workspace, tracked)
            streams.append(buffer.clone())
        else:
            streams.append(binding.compress_update(tracked, cur, nbits, tracked, buffer, workspace)[0].clone())
    s["streams"] = streams
    s["out"] = torch.empty_like(base)
    s["workspace"] = workspace if op == "merge" else binding.alloc_workspace(0, DEVICE)
    if op == "merge":
        s["stream"] = buffer.zero_()
    return s


def run(s):
    op = s["op"]
    if op == "compress":
        stream = binding.compress(s["base"], s["cur"], s["nbits"], s["stream"], s["workspace"])
        return s["stream"], stream.numel()  # `stream` is the part of the buffer that holds it
    if op == "snapshot":
        binding.compress_update_async(s["base"], s["cur"], s["nbits"], s["stream"], s["tracked"], s["workspace"])
        return s["stream"], s["tracked"]
    if op == "layers_snapshot":
        streams, _ = binding.compress_segments(s["base"], s["cur"], s["seg"], s["nbits"], s["stream"], s["workspace"], s["tracked"])
        return streams, s["tracked"]
    if op == "layers_recover":
        return binding.recover_segments(s["base"], s["streams"], s["seg"], s["nbits"], s["out"], s["workspace"])
    if op == "merge":
        stream = binding.merge(s["base"], s["streams"], s["nbits"], s["stream"], s["out"], s["workspace"])
        return s["stream"], stream.numel(), s["out"]
    # a chain longer than one call takes goes on from what the first call recovered
    src, streams = s["base"], s["streams"]
    for i in range(0, len(streams), binding.MAX_CHAIN):
        src = binding.recover(src, streams[i : i + binding.MAX_CHAIN], s["out"], s["workspace"])
    return src


def _stream_bytes(n, nbits):
    """About what a stream takes: three quarters of the nbits bits that a bucket index has, and the two indices."""
    return 0.75 * nbits * n / 8 + 72 * math.ceil(n / 4096) + 64 + 16 * 2 ** nbits


def work(case):
    op, n = case["op"], case["n"]
    stream = _stream_bytes(n, case["nbits"])
    k = case.get("k", 1)
    moved = {
        "compress": 8 * n + stream,
        "snapshot": 12 * n + stream,
        "layers_snapshot": 12 * n + stream,
        "recover": 8 * n + k * stream,
        "layers_recover": 8 * n + k * stream,
        "merge": 8 * n + (k + 1) * stream,  # base in, recovered state out, the merged stream out
    }[op]
    return {"bytes": moved, "flops": n * (k + 1)}


def tolerance(case):
    return "exact"
