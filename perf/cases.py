"""The work this library is measured by: chains of local operators through the package's entry points.

A case names a workload family of ``lop_inputs``, its sizes, its storage type, the number of row bands and how the chain
is called:

  resident       the input is on the device, all bands of every segment run (DeviceChain.run_banded)
  streamed       the input bands come from pinned host memory while earlier ones are computed (DeviceChain.run_pipelined)
  host_to_host   streamed, and the last layer stores the result into pinned host memory
  whole          every layer over all its rows (DeviceChain.run_whole)
  static         the entry point that allocates nothing (Plan.run_whole_static)

Weights, batch-norm scale / shift and inputs follow the recipe of ``lop_inputs`` (He-initialised weights, scale around
one, shift around zero, images uniform); they are drawn on the GPU from the seed because there are many millions of them.
"""
import math

import torch

import lop_inputs as li
import paper_2507_05829_b200 as lop
from lop_inputs import workloads as wk
from paper_2507_05829_b200.chain import DeviceChain


def listed():
    return [
        # the smallest call: one 3x3 convolution in fp32, four bands; launches and latency are all there is
        {"name": "conv_fp32", "family": "single_conv", "mode": "resident", "dtype": "f32", "n": 1, "h": 32, "w": 32, "c": 16, "bands": 4},
        # the same layer fed from host memory, as a device hands its input over band by band
        {"name": "conv_fp32_streamed", "family": "single_conv", "mode": "streamed", "dtype": "f32", "n": 1, "h": 32, "w": 32, "c": 16, "bands": 4},
        # one camera frame through the first block of a VGG, streamed
        {"name": "vgg_streamed", "family": "vgg_block", "mode": "streamed", "dtype": "bf16", "n": 1, "h": 224, "w": 224, "c": 64, "bands": 8},
        # the same block in full precision on an odd crop
        {"name": "vgg_fp32_odd", "family": "vgg_block", "mode": "resident", "dtype": "f32", "n": 1, "h": 181, "w": 203, "c": 64, "bands": 8},
        # a caller that must not allocate: the block inside another application's memory budget
        {"name": "vgg_static", "family": "vgg_block", "mode": "static", "dtype": "bf16", "n": 1, "h": 224, "w": 224, "c": 64, "bands": 1},
        # single-image classification, latency bound: the ResNet-18 trunk, streamed
        {"name": "resnet18_streamed", "family": "resnet18", "mode": "streamed", "dtype": "bf16", "n": 1, "h": 224, "w": 224, "c": 64, "bands": 8},
        # a few frames of an odd aspect ratio already on the device
        {"name": "resnet18_odd", "family": "resnet18", "mode": "resident", "dtype": "bf16", "n": 3, "h": 161, "w": 243, "c": 64, "bands": 5},
        # the headline: ResNet-50 trunk, batch 8, streamed
        {"name": "resnet50_streamed", "family": "resnet50", "mode": "streamed", "dtype": "bf16", "n": 8, "h": 224, "w": 224, "c": 64, "bands": 16},
        # the largest: a throughput batch of 32 on the device
        {"name": "resnet50_batch32", "family": "resnet50", "mode": "resident", "dtype": "bf16", "n": 32, "h": 224, "w": 224, "c": 64, "bands": 16},
        # a high-resolution detector backbone, host memory in and out
        {"name": "csp_host_to_host", "family": "csp_stack", "mode": "host_to_host", "dtype": "bf16", "n": 1, "h": 1024, "w": 1024, "c": 32, "bands": 32},
        # one ConvNeXt block: depth-wise 7x7, layer normalisation, point-wise MLP with GELU, shortcut
        {"name": "convnext", "family": "convnext_block", "mode": "resident", "dtype": "bf16", "n": 2, "h": 56, "w": 56, "c": 128, "bands": 8},
        # one DenseNet layer: 1x1, 3x3, concatenation; small maps
        {"name": "dense_layer", "family": "dense_layer", "mode": "resident", "dtype": "bf16", "n": 2, "h": 28, "w": 28, "c": 64, "bands": 4},
    ]


def _log(rng, lo, hi):
    """A whole number from lo to hi, spread over its logarithm."""
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    family = rng.choice(["single_conv", "vgg_block", "vgg_block", "resnet18", "resnet50", "csp_stack", "convnext_block", "pointwise_mlp", "dense_layer"])
    mode, dtype = rng.choice(["resident", "streamed", "host_to_host"]), "bf16"
    if family == "single_conv":
        dtype, n, c = "f32", rng.randint(1, 2), rng.choice([8, 16, 24, 32])
        h, w, bands = _log(rng, 16, 160), _log(rng, 16, 160), rng.randint(1, 8)
    elif family == "vgg_block":
        dtype, c = rng.choice(["bf16", "f32"]), 64
        mode = rng.choice(["resident", "streamed", "static"])
        h, w, bands = _log(rng, 48, 224), _log(rng, 48, 224), rng.randint(1, 12)
        if mode == "static":
            n, bands = 1, 1
            if dtype == "f32":                                  # its tensors take twice the built-in scratch
                h, w = min(h, 160), min(w, 160)
        else:
            n = rng.randint(1, 4)
    elif family in ("resnet18", "resnet50"):
        n, c = _log(rng, 1, 24), 64
        h, w, bands = rng.randint(96, 256), rng.randint(96, 256), rng.choice([4, 8, 16])
    elif family == "csp_stack":
        n, c = 1, 32
        h, w, bands = _log(rng, 256, 1152), _log(rng, 256, 1152), rng.choice([8, 16, 32])
    elif family == "dense_layer":
        n, c = rng.randint(1, 8), 32 * rng.randint(2, 12)
        h, w, bands = rng.randint(7, 56), rng.randint(7, 56), rng.randint(1, 6)
    else:
        mode = rng.choice(["resident", "streamed", "whole"])
        n, c = rng.randint(1, 8), rng.choice([64, 96, 128, 192, 256, 384])
        h, w, bands = _log(rng, 7, 96), _log(rng, 7, 96), rng.randint(1, 8)
    return {"family": family, "mode": mode, "dtype": dtype, "n": n, "h": h, "w": w, "c": c, "bands": bands}


def _workload(case):
    """The case's layer list and shapes, without data."""
    kw = dict(N=case["n"], H=case["h"], W=case["w"], n_bands=case["bands"], dtype=case["dtype"])
    family, c = case["family"], case["c"]
    if family in ("vgg_block", "resnet18", "resnet50"):
        kw["width"] = c
    elif family == "csp_stack":
        kw["base"] = c
    else:
        kw["C"] = c
        if family == "pointwise_mlp":
            kw["hidden"] = 4 * c
    return li.build(family, with_data=False, **kw)


def _has_weight(layer):
    return layer.op in (wk.CONV, wk.LINEAR, wk.DWCONV)


def prepare(case, seed):
    wl = _workload(case)
    gen = torch.Generator(device="cuda").manual_seed(seed)

    def normal(shape, mean, std):
        return (torch.randn(shape, generator=gen, device="cuda") * std + mean).cpu().numpy()

    for seg in wl.segments:
        for l in seg.layers:
            if _has_weight(l):
                cin = 1 if l.op == wk.DWCONV else l.cin
                l.weight = normal((l.cout, l.kh, l.kw, cin), 0.0, math.sqrt(2.0 / (l.kh * l.kw * cin)))
            if l.op == wk.LAYERNORM or (_has_weight(l) and wl.affine):
                l.scale, l.shift = normal((l.cout,), 1.0, 0.1), normal((l.cout,), 0.0, 0.1)
    lo, hi = wl.input_range
    x = (torch.rand((wl.N, wl.H, wl.W, wl.C), generator=gen, device="cuda") * (hi - lo) + lo).cpu().numpy()
    chain = DeviceChain(wl, flags=lop.LOP_FLAG_REUSE_HALO)
    state = {"mode": case["mode"], "chain": chain}
    if case["mode"] in ("streamed", "host_to_host"):
        state["x"] = chain.pinned_input(x)
    else:
        state["x"] = chain.input_tensor(x)
    if case["mode"] == "host_to_host":
        state["out"] = torch.empty(chain.outs[-1].shape, dtype=chain.outs[-1].dtype).pin_memory()
    if case["mode"] == "static":
        state["status"] = torch.zeros(1, dtype=torch.int32, device="cuda")
    return state


def run(state):
    chain, x, mode = state["chain"], state["x"], state["mode"]
    if mode == "resident":
        return chain.run_banded(x)
    if mode == "streamed":
        return chain.run_pipelined(x)
    if mode == "host_to_host":
        return chain.run_pipelined(x, out_pinned=state["out"])
    if mode == "whole":
        return chain.run_whole(x)
    out, status = chain.outs[0], state["status"]
    chain.plans[0].run_whole_static(x.data_ptr(), out.data_ptr(), status.data_ptr(), torch.cuda.current_stream().cuda_stream)
    return out, status


def _window(size, k, s, p, d):
    return (size + 2 * p - d * (k - 1) - 1) // s + 1


def work(case):
    """The chain's input, parameters and output once, and the multiply-adds of its layers."""
    wl = _workload(case)
    es = 2 if case["dtype"] == "bf16" else 4
    h, w, c = wl.H, wl.W, wl.C
    nbytes, flops = wl.N * h * w * c * es, 0
    for seg in wl.segments:
        shapes = {-1: (h, w)}
        for i, l in enumerate(seg.layers):
            hi, wi = shapes[l.input_from]
            ho, wo = _window(hi, l.kh, l.sh, l.ph, l.dh), _window(wi, l.kw, l.sw, l.pw, l.dw)
            shapes[i] = (ho, wo)
            pixels = wl.N * ho * wo
            if _has_weight(l):
                cin = 1 if l.op == wk.DWCONV else l.cin
                nbytes += l.cout * l.kh * l.kw * cin * es
                flops += 2 * pixels * l.cout * l.kh * l.kw * cin
            if l.op == wk.LAYERNORM or (_has_weight(l) and wl.affine):
                nbytes += 2 * l.cout * 4
            if l.op == wk.LAYERNORM:
                flops += 8 * pixels * l.cout                    # two sums, two subtractions, a square, a scale and a shift
        h, w = shapes[len(seg.layers) - 1]
        c = seg.layers[-1].cout
    return {"bytes": nbytes + wl.N * h * w * c * es, "flops": flops}


def tolerance(case):
    """fp32 sums of a few hundred to a few thousand products; or bf16 values, rounded once at every layer."""
    return {"rel": 1e-5} if case["dtype"] == "f32" else {"rel": 1e-2}
