"""Workloads on which the speed of the frame update is measured.

A case is one rollout of a batch of frame sequences through the public binding (`Graph`), from frame 0 on: a whole
clip at once (`rollout`), frame by frame as frames arrive (`step`), or in deep windows (`rollout_window`).  The
networks are the repository's own (`workloads.graphs`); weights are random with the variance the workloads use,
frames are a static image per sequence plus fresh noise on every frame, as in the paper's data (Sec. 4, Table A1).

Keys of a case:
  net      a network of `workloads.graphs.BUILDERS`, or "mnist" (the paper's MNIST network SR)
  size     image side of the input (0: the network's own)
  batch    sequences rolled out side by side
  frames   frame updates per pass
  pattern  rollout pattern: "streaming", "sequential" or "hybrid..."
  dtype    "bf16" or "fp32" states
  api      "run", "step" or "window" (then `frames` is a multiple of `window`)
  window   frames per deep window (0 otherwise)
  graphs   frames per CUDA graph (0: plain launches)
  states   whether the pass also hands out every node's state, as a program does that will resume the rollout later
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1806_04965_b200 import Graph
from workloads import data
from workloads import graphs as nets

DEVICE = "cuda:0"

# standard deviation of the per-frame noise, and whether the static image is uniform in [0, 1) or standard normal
NOISE = {"c1": (0.1, True), "c2": (0.3, True), "mnist": (0.3, True), "c3": (0.5, False), "c4": (0.2, True), "c4ff": (0.2, True),
         "c5": (1.0, False)}
# weight variance x fan-in: below 2 for the ReLU networks, so that rollouts with recurrence stay bounded at any length, as
# trained networks do
GAIN = 1.5


def _case(name, net, batch, frames, pattern="streaming", dtype="bf16", api="run", size=0, window=0, graphs=0, states=False):
    return {"name": name, "net": net, "size": size, "batch": batch, "frames": frames, "pattern": pattern, "dtype": dtype, "api": api,
            "window": window, "graphs": graphs, "states": states}


def listed():
    return [
        # the 784-128-128-10 perceptron in fp32 on a handful of short clips: almost no work, all launch and latency
        _case("mlp_b8", "c1", 8, 16, dtype="fp32"),
        # the same network in a control loop: one sequence, every frame its own call, levels evaluated inside the frame
        _case("mlp_b1_steps", "c1", 1, 16, pattern="sequential", dtype="fp32", api="step"),
        # small grey-image CNN with a skip and a recurrence on a batch of clips
        _case("cnn_b64", "c2", 64, 32),
        # the sequential rollout it is compared with, on what is left of a data set: an odd batch, states kept for later
        _case("cnn_b37_seq", "c2", 37, 20, pattern="sequential", states=True),
        # the paper's MNIST network SR in fp32 (validation against bf16), a batch of 100
        _case("mnist_fp32_b100", "mnist", 100, 12, dtype="fp32"),
        # the paper's CIFAR10 network with two added layers, live: one sequence, one call per frame (response time)
        _case("dsr2_b1_steps", "dsr2", 1, 16, api="step"),
        # the paper's deepest CIFAR10 network, evaluated on a batch of clips, states kept for the next window
        _case("dsr6_b128", "dsr6", 128, 16, graphs=16, states=True),
        # six-node network on 32 x 32 colour clips, a large batch, states kept for the next window
        _case("six_b256", "c3", 256, 20, states=True),
        # the same network as a two-stage pipeline on another image size and an odd batch, states kept for later
        _case("six_b37_hybrid", "c3", 37, 9, pattern="hybrid", size=28, states=True),
        # ten-node network with pooling edges and 43 classes, long clips, states kept for the next window
        _case("ten_b128", "c4", 128, 64, graphs=16, states=True),
        # the same network without recurrence: first frames of a clip classified side by side in deep windows
        _case("ten_window8_b128", "c4ff", 128, 16, pattern="sequential", api="window", window=8, states=True),
        # sixteen 128-channel nodes on 64 x 64 clips with random skips and recurrences: the largest work
        _case("stress_b32", "c5", 32, 128, states=True),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    net = rng.choice(["c1", "c1", "c2", "c2", "mnist", "dsr2", "dsr4", "dsr6", "c3", "c3", "c4", "c4ff", "c5"])
    c = _case("", net, 1, 1)
    del c["name"]
    # largest batch, frames, image sizes, data types
    b_max, f_max, sizes, dtypes = {
        "c1": (256, 64, [0], ["fp32", "fp32", "bf16"]),
        "c2": (256, 64, [0], ["bf16", "bf16", "bf16", "fp32"]),
        "mnist": (256, 32, [0], ["fp32", "bf16"]),
        "dsr2": (256, 32, [0], ["bf16"]), "dsr4": (256, 32, [0], ["bf16"]), "dsr6": (256, 32, [0], ["bf16"]),
        "c3": (256, 32, [16, 20, 24, 28, 32, 32, 36, 40], ["bf16"]),
        "c4": (128, 64, [16, 20, 24, 28, 32, 32, 36, 40], ["bf16"]),
        "c4ff": (128, 32, [16, 20, 24, 28, 32, 32, 36, 40], ["bf16"]),
        "c5": (32, 64, [32, 40, 48, 64, 64], ["bf16"]),
    }[net]
    c["size"], c["dtype"] = rng.choice(sizes), rng.choice(dtypes)
    c["batch"], c["frames"] = _log_int(rng, 1, b_max), _log_int(rng, 4, f_max)
    if c["dtype"] == "fp32" and net != "c1":                 # CUDA-core arithmetic: the work stays that of a check
        c["batch"] = min(c["batch"], 128)
        c["frames"] = min(c["frames"], 16)
    c["pattern"] = rng.choice(["streaming", "streaming", "sequential"] + {"c3": ["hybrid"], "c5": ["hybrid0", "hybrid1"]}.get(net, []))
    c["api"] = "step" if c["batch"] <= 8 and rng.random() < 0.7 else "run"
    if net == "c4ff":
        c["pattern"], c["api"] = "sequential", rng.choice(["window", "window", "run"])
    if c["api"] == "window":
        c["window"] = rng.choice([2, 4, 8])
        c["frames"] = max(1, c["frames"] // c["window"]) * c["window"]
        c["batch"] = min(c["batch"], 128)
    if c["api"] == "run":
        c["graphs"] = rng.choice([0, 0, 4, 16])
        c["states"] = rng.random() < 0.3
    return c


def _spec(case):
    over = dict(batch=case["batch"], frames=case["frames"])
    if case["size"]:
        over["size"] = case["size"]
    if case["net"] == "mnist":
        g = nets.mnist_net("SR", **over)
        g.dtype = case["dtype"]
        nets.check_shapes(g)
        return g
    g = nets.build(case["net"], **over)
    g.dtype = case["dtype"]
    return g


def prepare(case, seed):
    spec = _spec(case)
    gen = torch.Generator(device=DEVICE).manual_seed(int(seed))
    fan = [0] * len(spec.nodes)
    for ei, e in enumerate(spec.edges):
        fan[e.tgt] += data.edge_fan_in(spec, ei)
    graph = Graph(spec.nodes, spec.edges, spec.patterns[case["pattern"]], batch=spec.batch, dtype=spec.dtype, graph_frames=case["graphs"],
                  device=DEVICE)
    weights = []
    for ei, e in enumerate(spec.edges):
        w = torch.randn(data.weight_shape(spec, ei), generator=gen, device=DEVICE) * math.sqrt(min(GAIN, spec.weight_gain) / fan[e.tgt])
        weights.append(w.cpu().numpy())
    biases = [0.05 * torch.randn(v.c, generator=gen, device=DEVICE).cpu().numpy().astype(np.float32) for v in spec.nodes]
    graph.set_weights(weights, biases)
    if case["api"] == "window":
        graph.bind_window(case["window"])
    sigma, uniform = NOISE.get(case["net"], (0.3, True))
    frames = []
    for v in graph.input_nodes:
        n = spec.nodes[v]
        shape = (spec.batch, n.h, n.w, n.c)
        base = (torch.rand if uniform else torch.randn)(shape, generator=gen, device=DEVICE)
        x = torch.empty((spec.frames + 1,) + shape, dtype=graph.tdtype, device=DEVICE)
        for t in range(spec.frames + 1):
            x[t] = base + sigma * torch.randn(shape, generator=gen, device=DEVICE)
        frames.append(x)
    return {"graph": graph, "frames": frames, "T": spec.frames, "api": case["api"], "window": case["window"], "states": case["states"]}


def run(state):
    graph, frames, T = state["graph"], state["frames"], state["T"]
    if state["api"] == "run":
        out = graph.rollout(frames)
    else:
        out = torch.empty((T,) + graph.out_shape(), dtype=torch.float32, device=DEVICE)
        graph.reset([f[0] for f in frames])
        if state["api"] == "step":
            for t in range(T):
                graph.step([f[t + 1] for f in frames], out[t])
        else:
            for t in range(0, T, state["window"]):
                graph.rollout_window([f[t + 1:t + 1 + state["window"]] for f in frames], out[t:t + state["window"]])
    if not state["states"]:
        return out
    return [out] + [graph.get_state(v) for v in range(len(graph.nodes)) if v not in graph.input_nodes]


def work(case):
    """Input frames and weights read once, outputs (and states, where they are asked for) written once; the
    multiply-adds of every edge at every frame."""
    spec = _spec(case)
    el = 4 if spec.dtype == "fp32" else 2
    ins = spec.input_nodes()
    n_bytes = (spec.frames + 1) * spec.batch * el * sum(spec.nodes[v].h * spec.nodes[v].w * spec.nodes[v].c for v in ins)
    n_bytes += el * sum(int(np.prod(data.weight_shape(spec, ei))) for ei in range(len(spec.edges)))
    out = spec.nodes[-1]
    n_bytes += spec.frames * spec.batch * 4 * out.h * out.w * out.c
    if case["states"]:
        n_bytes += spec.batch * el * sum(n.h * n.w * n.c for v, n in enumerate(spec.nodes) if v not in ins)
    return {"bytes": n_bytes, "flops": 2 * nets.macs_per_sample(spec) * spec.batch * spec.frames}


def tolerance(case):
    """fp32: sums of up to a few thousand terms in another order.  bf16: states are rounded to bf16 on every frame, and
    a sum in another order rounds some of them the other way; the differences run through every layer and, with
    recurrence, through every frame."""
    if case["dtype"] == "fp32":
        return {"rel": 5e-6, "max": 5e-5}
    return {"rel": 2e-2, "max": 2e-1}
