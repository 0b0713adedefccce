"""Performance cases of the COMP-AMS optimizer: the steps that training programs have it do.

A case is one optimizer step in the middle of a run: the handle exists, its error accumulators and moments are
those of a run that has been going for a while, and a fresh gradient batch lies on the GPU. listed() names the cases
that are followed; draw() gives others of the same ranges: 1 to 32 workers, 2^16 to 2^27 parameters of any
remainder, the whole vector or many tensors as blocks, the four kinds of step (Top-k, Block-Sign, Random-k,
uncompressed), kept shares from 0.1 % to 10 %, fp32 and bfloat16 gradients, and the three ways of calling: step()
on an [n, d] gradient tensor, the optimizer of a torch model, and compress() / apply() of one rank of a sharded job.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

from paper_2205_05632_b200 import BLOCKSIGN, RANDK, TOPK, CompAMS
from paper_2205_05632_b200 import workloads as W
from paper_2205_05632_b200.optim import CompAMSOptimizer

COMPRESSOR = {"topk": TOPK, "sign": BLOCKSIGN, "randk": RANDK, "dense": TOPK}
WARM_STEPS = 40  # steps a handle has done before the measured one: the accumulators fill, the thresholds settle
WINDOW = 64      # elements between two windows of a gradient buffer: 256 bytes in fp32, 128 in bfloat16
WINDOWS = 64


def case(name, entry, kind, blocks, n, d, ratio=0.01, dtype="f32", layers=0, n_total=0):
    c = {"entry": entry, "kind": kind, "blocks": blocks, "n": n, "d": d, "ratio": ratio, "dtype": dtype,
         "layers": layers, "n_total": n_total}
    if name:
        c["name"] = name
    return c


RESNET18 = int(W.offsets_from_shapes(W.resnet18_cifar_shapes())[-1])
RESNET50 = int(W.offsets_from_shapes(W.resnet50_imagenet_shapes())[-1])


def listed():
    return [
        # a small model or a single layer: latency and launches are what a step costs
        case("small topk n=4 d=65536", "step", "topk", "whole", 4, 65536),
        # a small model with the sign compressor; everything fits the L2 cache
        case("small sign n=8 d=2^20", "step", "sign", "whole", 8, 1 << 20),
        # the usual data-parallel job on a CIFAR-sized network, per-tensor signs
        case("resnet18 sign n=16", "step", "sign", "resnet18", 16, RESNET18),
        # the same network with the paper's compressor over the whole vector, at the sparser of its two ratios
        case("resnet18 topk 0.1% n=16", "step", "topk", "resnet18-whole", 16, RESNET18, ratio=0.001),
        # mixed-precision training: bfloat16 gradients
        case("resnet18 topk 1% bf16 n=16", "step", "topk", "resnet18-whole", 16, RESNET18, dtype="bf16"),
        # an ImageNet-sized network on 32 workers, layer-wise selection
        case("resnet50 topk layerwise n=32", "step", "topk", "resnet50", 32, RESNET50),
        # random sparsification
        case("resnet18 randk n=16", "step", "randk", "resnet18-whole", 16, RESNET18),
        # the uncompressed baseline every comparison with the compressors runs, ragged length
        case("dense n=8 d=16777213", "step", "dense", "whole", 8, 16777213, ratio=1.0),
        # a mild compression ratio: ten per cent of an odd-sized vector kept
        case("topk 10% n=8 d=4194301", "step", "topk", "whole", 8, 4194301, ratio=0.1),
        # the optimizer of a torch model: four micro-batches as workers, gradients collected tensor by tensor
        case("model resnet18 topk n=4", "model", "topk", "resnet18", 4, RESNET18),
        # one rank of a sharded job: 8 of 32 workers here, the other ranks' messages arrive between the two halves
        case("shard resnet50 sign 8 of 32", "shard", "sign", "resnet50", 8, RESNET50, n_total=32),
        # the largest step that one GPU is used for: 17 GB of gradients
        case("largest topk n=32 d=2^27", "step", "topk", "whole", 32, 1 << 27),
    ]


def draw(rng: random.Random):
    entry = rng.choices(["step", "model", "shard"], [10, 1, 1])[0]
    kind = rng.choices(["topk", "sign", "randk", "dense"], [5, 3, 1, 1])[0]
    if entry == "shard" and kind == "dense":
        kind = "topk"  # a sharded job exchanges compressed gradients
    n = int(round(math.exp(rng.uniform(0.0, math.log(32.0)))))
    d = int(math.exp(rng.uniform(math.log(2.0 ** 16), math.log(2.0 ** 27))))
    while n * d > 1 << 30:
        d = d // 2 + rng.randrange(64)
    if entry == "model":
        n, d = min(n, 8), min(d, 1 << 24)
    if rng.random() < 0.3:
        d -= d % 32  # padded parameter vectors are common, ragged ones more so
    layers = 0
    blocks = "whole"
    if entry == "model" or rng.random() < 0.5:
        blocks, layers = "layers", rng.randrange(4, 160)
    ratio = 1.0 if kind == "dense" else round(math.exp(rng.uniform(math.log(0.001), math.log(0.1))), 5)
    dtype = "bf16" if entry == "step" and rng.random() < 0.3 else "f32"
    n_total = n * rng.choice([2, 4]) if entry == "shard" else 0
    return case(None, entry, kind, blocks, n, d, ratio, dtype, layers, n_total)


def tensor_sizes(c):
    """Sizes of the parameter tensors, definition order."""
    if c["blocks"].startswith("resnet18"):
        return [W.numel(s) for s in W.resnet18_cifar_shapes()]
    if c["blocks"] == "resnet50":
        return [W.numel(s) for s in W.resnet50_imagenet_shapes()]
    if c["blocks"] == "layers":  # weights that grow with depth, each followed by a small bias
        g = np.random.default_rng(c["layers"] * 1000003 + c["d"])
        w = g.lognormal(0.0, 1.0, c["layers"]) * np.linspace(0.2, 2.0, c["layers"])
        w[1::2] *= 0.002
        sizes = np.maximum(1, np.floor(w / w.sum() * c["d"]).astype(np.int64))
        k = int(np.argmax(sizes))
        sizes[k] += c["d"] - int(sizes.sum())
        return [int(s) for s in sizes]
    return [c["d"]]


def offsets(c):
    if c["blocks"] in ("whole", "resnet18-whole"):
        return np.array([0, c["d"]], dtype=np.int64)
    return np.concatenate([[0], np.cumsum(tensor_sizes(c))]).astype(np.int64)


def gradients(c, gen, n):
    """Gradient batches [n, d], a different one for every step: whole vectors of N(0, 1) draws are windows that move
    over one buffer; where the value scale depends on the tensor, a ring of separate batches of Student-t values
    (df = 3, scaled by fan-in^-1/2, 5 % exact zeros)."""
    d = c["d"]
    dt = torch.bfloat16 if c["dtype"] == "bf16" else torch.float32
    if c["blocks"] == "whole":
        flat = torch.empty(n * d + WINDOW * WINDOWS, device="cuda", dtype=dt)
        for lo in range(0, flat.numel(), 1 << 28):
            flat[lo:lo + (1 << 28)].normal_(generator=gen)
        return [flat[WINDOW * k:WINDOW * k + n * d].view(n, d) for k in range(WINDOWS)]
    if c["blocks"].startswith("resnet"):
        shapes = W.resnet50_imagenet_shapes() if c["blocks"] == "resnet50" else W.resnet18_cifar_shapes()
        scale = W.per_coordinate_scale(shapes, "cuda")
    else:
        sizes = torch.tensor(tensor_sizes(c), device="cuda")
        scale = torch.repeat_interleave(sizes.float().pow(-0.25), sizes)
    ring = []
    for _ in range(8 if n * d <= 1 << 28 else 4):
        G = torch.empty(n, d, device="cuda", dtype=dt)
        for i in range(n):
            g = W.student_t3(gen, d, "cuda") * scale
            g[torch.rand(d, generator=gen, device="cuda") < 0.05] = 0.0
            G[i] = g
        ring.append(G)
    return ring


class State:
    """A training program's optimizer, parameters and gradient batches."""


def prepare(c, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    s = State()
    s.case, s.t = c, 0
    n, d, comp = c["n"], c["d"], COMPRESSOR[c["kind"]]
    theta = 0.1 * torch.randn(d, generator=gen, device="cuda")
    batches = gradients(c, gen, n)
    if c["entry"] == "model":
        sizes = tensor_sizes(c)
        s.params = [torch.nn.Parameter(t) for t in torch.split(theta, sizes)]
        s.opt = CompAMSOptimizer(s.params, n, comp, c["ratio"], whole_vector=c["blocks"] == "whole", seed=seed)
        s.theta = s.opt.theta
        # what backward() leaves for every micro-batch: one tensor per parameter, each its own allocation
        s.batches = [[[t.clone() for t in torch.split(G[i], sizes)] for i in range(n)] for G in batches]
        handle = s.opt.opt
    else:
        s.theta, s.batches = theta, batches
        s.opt = handle = CompAMS(n, d, offsets(c), comp, c["ratio"], n_total=c["n_total"] or None)
        if c["kind"] == "randk":
            handle.set_seed(seed)
    s.arrived = None
    if c["entry"] == "shard":  # the messages of the other ranks' workers
        rest = CompAMS(c["n_total"] - n, d, offsets(c), comp, c["ratio"], n_total=c["n_total"], first_worker=n)
        if c["kind"] == "randk":
            rest.set_seed(seed)
        G = torch.cat([batches[k % len(batches)] for k in range(c["n_total"] // n - 1)])
        rest.compress(G)
        s.arrived = [b[n:].clone() for b in rest.message_buffers()]
        rest.close()
    s.moments = [handle.buffer(name) for name in ("m", "v", "vhat")]
    for _ in range(WARM_STEPS):
        run(s)
    return s


def run(s):
    """One optimizer step; the updated parameters and moments."""
    batch = s.batches[s.t % len(s.batches)]
    s.t += 1
    entry = s.case["entry"]
    if entry == "step":
        s.opt.step(batch, s.theta)
    elif entry == "model":
        for i, grads in enumerate(batch):
            for p, g in zip(s.params, grads):
                p.grad = g  # as the micro-batch's backward() leaves it
            s.opt.collect(i)
        s.opt.step()
    else:
        s.opt.compress(batch)
        for buf, theirs in zip(s.opt.message_buffers(), s.arrived):
            buf[s.case["n"]:].copy_(theirs)  # in place of the all-gather
        s.opt.apply(s.theta)
    return [s.theta] + s.moments


def work(c):
    """Bytes: every worker's gradient read, its error accumulator read and written (k = d keeps none), theta, m, v and
    vhat read and written. Operations per worker-element: the addition g + e, a comparison or absolute sum, the
    residual; per coordinate the average and the AMSGrad update (about 12)."""
    n, d = c["n"], c["d"]
    g = 2 if c["dtype"] == "bf16" else 4
    per_worker = g if c["kind"] == "dense" else g + 8
    return {"bytes": (per_worker * n + 32) * d, "flops": (3 * n + 12) * d}


def tolerance(c):
    """Kept sets and sign bits are exact, so what may differ is the rounding of fp32 values carried over the 41 steps
    behind an output. Against the server's sums and state in 64 bits: theta 1.6e-7 (largest 1.0e-6), m 9e-8 (7e-7),
    v and vhat 1.4e-7 (9e-7), for Top-k, Block-Sign and k = d alike; about four times that is allowed."""
    return {"rel": 7e-7, "max": 5e-6}
