"""The work whose speed counts: whole inferences through the public entry points, over the range of networks, batches,
image sizes and calling styles that a user of the executor has.

A case is one network at one batch and image size, run under the plan the auto-tuner proposes (what the README and the
benchmark tell a user to install), in one of three calling styles:

  device   the input is already on the GPU; one asynchronous `dlf_net_run` on the current stream (the benchmark's step, and
           what a pipeline with its own device buffers does);
  host     one `dlf_net_run_host` on page-locked host buffers: copy in, run, copy out, wait (the end-to-end call);
  serve    the Python loop over batches that arrive in host memory: `Session.upload`, `Session.run`, the result read back -
           every batch in a device tensor of its own, as the loop in a script would have it.

Weights are in host arrays and go through `Session`, drawn on the GPU from the seed with the distributions of the
repository's workload recipe: activations U(-1, 1), weights N(0, 1/fan_in), biases N(0, 0.01).
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2011_05630_b200 import binding as B
from paper_2011_05630_b200 import networks as nw
from paper_2011_05630_b200 import plans
from paper_2011_05630_b200.runtime import Session

# Classifiers of the repository's benchmark: builder, largest batch it is run at there, the image sizes it takes (networks
# that end in fully connected layers over a flattened map take 224 x 224 alone).
_NETS = {
    "resnet50": (nw.resnet50, 32, True),
    "resnet18": (nw.resnet18, 32, True),
    "mobilenet_v2": (nw.mobilenet_v2, 64, True),
    "vgg16": (nw.vgg16, 8, False),
    "vgg19": (nw.vgg19, 8, False),
    "alexnet": (nw.alexnet, 32, False),
}
_MAX_FLOPS = 4.8e11         # of a drawn case: as many as the largest listed one has
_MAX_CHAIN_BYTES = 160e6    # all maps of a drawn chain: a little more than the largest listed one's
_SERVE_BATCHES = 3          # batches that one pass of the serving loop works off


def listed():
    net = lambda name, arch, n, h, w, mode: {"name": name, "kind": "net", "net": arch, "n": n, "h": h, "w": w, "mode": mode}
    chain = lambda name, depth, c, k, n, h, w: {"name": name, "kind": "chain", "depth": depth, "c": c, "k": k, "n": n, "h": h,
                                               "w": w, "mode": "device"}
    return [
        # the smallest fusion group: two 3x3 16 -> 16 layers on one 32 x 32 image; launch latency is all there is
        chain("two_layer_b1", 2, 16, 3, 1, 32, 32),
        # a run of narrow 3x3 layers on an odd-sized map and an odd batch, as a detector's or a denoiser's trunk has it
        chain("chain4_c64_27x29_b5", 4, 64, 3, 5, 27, 29),
        # the heavy end of the characterisation sweep: wide 3x3 layers on a large map, bound by the tensor cores
        chain("chain2_c512_56x56_b16", 2, 512, 3, 16, 56, 56),
        # one image at a time (interactive classification): latency of 56 layers
        net("resnet50_b1", "resnet50", 1, 224, 224, "device"),
        # throughput classification, the benchmark's default workload
        net("resnet50_b32", "resnet50", 32, 224, 224, "device"),
        # a batch that arrives uncropped: sizes that divide evenly by nothing
        net("resnet50_b6_203x261", "resnet50", 6, 203, 261, "device"),
        # the same throughput workload end to end from page-locked host buffers
        net("resnet50_b32_host", "resnet50", 32, 224, 224, "host"),
        # batches served one after another from a Python loop
        net("resnet18_b8_serve", "resnet18", 8, 224, 224, "serve"),
        # large 3x3 layers with fused pooling and three fully connected layers that stream their weights
        net("vgg16_b8", "vgg16", 8, 224, 224, "device"),
        # 11x11 and 5x5 kernels, overlapping pools
        net("alexnet_b32", "alexnet", 32, 224, 224, "device"),
        # depthwise and narrow pointwise layers: one image, where launches count, and a large batch, where bytes count
        net("mobilenet_v2_b1", "mobilenet_v2", 1, 224, 224, "device"),
        net("mobilenet_v2_b64", "mobilenet_v2", 64, 224, 224, "device"),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    while True:
        if rng.random() < 0.3:
            h = _log_int(rng, 7, 112)
            case = {"kind": "chain", "depth": rng.randint(1, 8), "c": rng.choice([16, 24, 32, 64, 96, 128, 256, 512]),
                    "k": rng.choice([1, 3, 3]), "n": _log_int(rng, 1, 16), "h": h, "w": max(7, min(112, h + rng.randint(-3, 3))),
                    "mode": "device"}
        else:
            arch = rng.choice(sorted(_NETS))
            _, max_batch, any_size = _NETS[arch]
            h = w = 224
            if any_size and rng.random() < 0.6:
                h, w = rng.randint(128, 288), rng.randint(128, 288)
            n = _log_int(rng, 1, max(1, min(max_batch, max_batch * 224 * 224 // (h * w))))
            case = {"kind": "net", "net": arch, "n": n, "h": h, "w": w,
                    "mode": rng.choice(["device", "device", "host"] + (["serve"] if n <= 8 else []))}
        # no heavier than the largest listed ones: in operations, and in the bytes of a chain's maps
        maps = 2 * (case["depth"] + 1) * case["n"] * case["h"] * case["w"] * case["c"] if case["kind"] == "chain" else 0
        if maps <= _MAX_CHAIN_BYTES and work(case)["flops"] <= _MAX_FLOPS:
            return case


def _layers(case):
    if case["kind"] == "chain":
        return nw.conv_chain(case["depth"], case["c"], case["k"]), case["c"]
    return _NETS[case["net"]][0](), 3


def _params(layers, gen):
    """Weights [cout][kh][kw][cin/groups] fp16 and biases fp32, in host memory as `Session` takes them."""
    out = []
    for l in layers:
        if l["op"] in ("conv", "dwconv"):
            cg = l["cin"] // l["groups"]
            shape, fan = (l["cout"], l["kh"], l["kw"], cg), l["kh"] * l["kw"] * cg
        elif l["op"] == "fc":
            shape, fan = (l["cout"], l["cin"]), l["cin"]
        else:
            out.append(None)
            continue
        w = torch.randn(shape, generator=gen, device="cuda").mul_(fan ** -0.5).half().cpu().numpy()
        b = torch.randn((l["cout"],), generator=gen, device="cuda").mul_(0.1).cpu().numpy()
        out.append((w, b))
    return out


def prepare(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    layers, c = _layers(case)
    n, h, w = case["n"], case["h"], case["w"]
    sess = Session(layers, _params(layers, gen), n, h, w, c)
    sess.set_plan(*plans.tuned_plan(sess.net, len(layers)))
    image = lambda: (torch.rand((n, h, w, c), generator=gen, device="cuda") * 2.0 - 1.0).half()
    state = {"mode": case["mode"], "sess": sess}
    if case["mode"] == "device":
        state["x"] = image()
    elif case["mode"] == "host":
        state["x"] = image().cpu().pin_memory()
        state["y"] = torch.empty(sess.out_shape, dtype=torch.float16, pin_memory=True)
    else:
        state["batches"] = [image().cpu().numpy() for _ in range(_SERVE_BATCHES)]
    return state


def run(state):
    sess = state["sess"]
    if state["mode"] == "device":
        B.net_run(sess.net, state["x"].data_ptr(), sess.out.data_ptr(), torch.cuda.current_stream().cuda_stream)
        return sess.out
    if state["mode"] == "host":
        B.net_run_host(sess.net, state["x"].data_ptr(), state["y"].data_ptr(), torch.cuda.current_stream().cuda_stream)
        return state["y"]
    results = []
    for batch in state["batches"]:
        x = sess.upload(batch)
        results.append(sess.run(x).cpu())
    return results


def work(case):
    """The network's input, weights and biases read once and its output written once (every map in between could stay on
    the chip); the useful operations of all its layers."""
    layers, c = _layers(case)
    n, h, w = case["n"], case["h"], case["w"]
    net = B.net_create(layers, n, h, w, c)
    try:
        info = [B.net_layer_info(net, i) for i in range(len(layers))]
    finally:
        B.net_destroy(net)
    flops = sum(fl for _, fl, _ in info)
    weights = 0
    for l in layers:
        if l["op"] in ("conv", "dwconv"):
            weights += l["cout"] * l["kh"] * l["kw"] * (l["cin"] // l["groups"]) * 2 + l["cout"] * 4
        elif l["op"] == "fc":
            weights += l["cout"] * l["cin"] * 2 + l["cout"] * 4
    maps = n * h * w * c * 2 + int(np.prod(info[-1][2])) * 2
    times = _SERVE_BATCHES if case["mode"] == "serve" else 1
    return {"bytes": times * (maps + weights), "flops": times * flops}


def tolerance(case):
    """fp16 maps with one rounding (2^-11 of a value) per layer, sums in fp32: layers in another order of summation differ
    by single roundings, which the following layers carry on.  Measured against the same layers with sums in 64 bits: up to
    2.1e-4 for the chains and 3.0e-4 .. 5.3e-4 for the networks, single values up to 3.3e-3 of the output's root mean
    square; about four times that."""
    return {"rel": 1e-3 if case["kind"] == "chain" else 2e-3, "max": 1.5e-2}
