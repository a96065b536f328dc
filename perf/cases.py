"""The work that programs have this library do, as cases that can be timed and compared.

Three kinds of call, all through the public entry points of the binding:

  net   squeezenet_forward (or, with "host", squeezenet_forward_host): SqueezeNet v1.0 on a batch of 227x227 images
  fire  fire_forward: one fire layer (squeeze, both expands)
  conv  conv_forward_ex: one convolution layer, with the fused pooling options where asked

in the three precisions the library has.  Sizes are the layer shapes of SqueezeNet and of the bottleneck network (the
second workload of the tests), the batches of the benchmark's sweeps, and generic odd ones.  Kernels are He-normal,
biases N(0, 0.01), images U[0,1), activations |N(0,1)|: what the tests and the benchmark draw, made on the device here.
"""
import math

import numpy as np
import torch

from paper_1611_07151_b200 import binding as B
from paper_1611_07151_b200 import synth

DTYPE = {"f32": B.SQN_F32, "bf16": B.SQN_BF16, "f16": B.SQN_F16}
TORCH = {"f32": torch.float32, "bf16": torch.bfloat16, "f16": torch.float16}
SIZE = {"f32": 4, "bf16": 2, "f16": 2}
IMG = 227
# (input layers, squeeze layers, layers of each expand, rows = columns) of fire2 .. fire9
FIRES = [(96, 16, 64, 55), (128, 16, 64, 55), (128, 32, 128, 55), (256, 32, 128, 27),
         (256, 48, 192, 27), (384, 48, 192, 27), (384, 64, 256, 27), (512, 64, 256, 13)]


def _net(name, dtype, batch, packed=False, host=False):
    return {"name": name, "kind": "net", "dtype": dtype, "batch": batch, "packed": packed, "host": host}


def _fire(name, dtype, batch, cin, s, e, h, w):
    return {"name": name, "kind": "fire", "dtype": dtype, "batch": batch, "cin": cin, "s": s, "e": e, "h": h, "w": w}


def _conv(name, dtype, batch, cin, cout, h, w, k, s=1, pad=0, pool="none"):
    return {"name": name, "kind": "conv", "dtype": dtype, "batch": batch, "cin": cin, "cout": cout, "h": h, "w": w, "k": k,
            "s": s, "pad": pad, "pool": pool}


def listed():
    return [
        # classifying one image as it arrives, on the exact path and on the fast one: launches and latencies count
        _net("net_f32_b1", "f32", 1),
        _net("net_bf16_b1", "bf16", 1),
        # a small batch collected by a server, of no round size, half precision
        _net("net_f16_b19", "f16", 19),
        # throughput on large batches: images resident on the device in the stem's offline layout; the exact path
        _net("net_bf16_b256_packed", "bf16", 256, packed=True),
        _net("net_f32_b256", "f32", 256),
        # images that arrive in host memory, results that are wanted there
        _net("net_bf16_b64_host", "bf16", 64, host=True),
        # one layer and one fire layer of one image: the smallest calls, exact path
        _conv("conv3x3_f32_16to64_55_b1", "f32", 1, 16, 64, 55, 55, 3, pad=1),
        _fire("fire4_f32_b1", "f32", 1, 128, 32, 128, 55, 55),
        # a fire layer whose kernels do not fit one SM, mixed precision, a batch of no round size
        _fire("fire8_bf16_b37", "bf16", 37, 384, 64, 256, 27, 27),
        # layers of another network through the single-layer entry point: the 3x3 of a bottleneck block, a wide 1x1
        _conv("conv3x3_bf16_256to256_14_b64", "bf16", 64, 256, 256, 14, 14, 3, pad=1),
        _conv("conv1x1_bf16_128to512_28_b17", "bf16", 17, 128, 512, 28, 28, 1),
        # the exact path takes any shape: stride, padding, ragged map and layer counts
        _conv("conv5x5s2_f32_20to36_61x47_b9", "f32", 9, 20, 36, 61, 47, 5, s=2, pad=2),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    dtype = rng.choice(["f32", "bf16", "bf16", "f16"])
    kind = rng.choice(["net", "fire", "conv", "conv"])
    if kind == "net":
        batch = _log_int(rng, 1, 256)
        host = rng.random() < 0.25
        packed = dtype == "bf16" and not host and rng.random() < 0.5
        c = _net("", dtype, batch, packed, host)
    elif kind == "fire":
        cin, s, e, hw = rng.choice(FIRES)
        h, w = (hw, hw) if rng.random() < 0.5 else (_log_int(rng, 7, 60), _log_int(rng, 7, 60))
        c = _fire("", dtype, _log_int(rng, 1, 256), cin, s, e, h, w)
    else:
        shape = rng.choice(["squeezenet", "bottleneck", "generic"])
        if shape == "generic":
            # the tensor-core paths take stride 1 and layer counts in steps of 16, the exact path anything
            step = 1 if dtype == "f32" else 16
            k = rng.choice([1, 2, 3, 3, 5] if dtype == "f32" else [1, 3, 3, 5])
            cin, cout = (step * _log_int(rng, 1, 256 // step) for _ in range(2))
            h, w = (_log_int(rng, 7, 80) for _ in range(2))
            c = _conv("", dtype, _log_int(rng, 1, 32), cin, cout, h, w, k, s=rng.choice([1, 2]) if dtype == "f32" else 1,
                      pad=k // 2)
        else:
            table = synth.SQUEEZENET_CONVS if shape == "squeezenet" else synth.BOTTLENECK_CONVS
            _, cin, cout, k, s, pad, hw = rng.choice(table)
            c = _conv("", dtype, _log_int(rng, 1, 128), cin, cout, hw, hw, k, s=s, pad=pad)
            if dtype != "f32" and c["k"] == 7 and rng.random() < 0.5:
                c["pool"] = "max"
            if dtype != "f32" and c["cout"] == 1000 and rng.random() < 0.5:
                c["pool"] = "avg"
    del c["name"]
    return c


# ------------------------------------------------------------------------------------------------------- inputs
def _params(gen, dtype, cout, k, cin):
    """He-normal kernels [cout][k][k][cin] in the path's type and an fp32 bias."""
    w = torch.randn((cout, k, k, cin), generator=gen, device="cuda") * math.sqrt(2.0 / (cin * k * k))
    b = torch.randn((cout,), generator=gen, device="cuda") * 0.01
    return w.to(TORCH[dtype]), b


def _activations(gen, dtype, shape):
    return torch.randn(shape, generator=gen, device="cuda").abs_().to(TORCH[dtype])


def _net_state(case, gen):
    dtype, batch = case["dtype"], case["batch"]
    params = [_params(gen, dtype, cout, k, cin) for _, cin, cout, k, _, _, _ in synth.SQUEEZENET_CONVS]
    weights, biases = [w for w, _ in params], [b for _, b in params]
    images = torch.rand((batch, IMG, IMG, 3), generator=gen, device="cuda").to(TORCH[dtype])
    if case["packed"]:
        # the stem's offline layouts: kernels through the library's helper, images padded to [228][228][4] with ones in
        # the fourth layer of every image pixel
        hp, wp = B.sqn_stem_packed_extent(IMG, IMG)
        packed = torch.zeros((batch, hp, wp, 4), dtype=torch.bfloat16, device="cuda")
        packed[:, :IMG, :IMG, :3] = images
        packed[:, :IMG, :IMG, 3] = 1.0
        images = packed
        first = weights[0].float().permute(0, 3, 1, 2).cpu().numpy()
        weights[0] = B.to_device(B.sqn_pack_stem_weights(first, biases[0].cpu().numpy()), B.SQN_BF16)
    net = B.squeezenet_create(weights, biases, DTYPE[dtype], batch)
    if case["packed"]:
        B.squeezenet_set_stem_prepacked(net)
    if case["host"]:
        nbytes = B.squeezenet_host_workspace_bytes(net, batch)
        images = images.cpu().pin_memory()
        outs = [torch.zeros((batch, 1000)).pin_memory() for _ in range(2)]
    else:
        nbytes = B.squeezenet_workspace_bytes(net, batch)
        outs = [torch.zeros((batch, 1000), device="cuda") for _ in range(2)]
    return {"net": net, "keep": (weights, biases), "images": images, "outs": outs,
            "work": torch.empty(nbytes, dtype=torch.uint8, device="cuda")}


def _fire_state(case, gen):
    dtype = case["dtype"]
    cin, s, e, h, w, batch = (case[k] for k in ("cin", "s", "e", "h", "w", "batch"))
    params = [_params(gen, dtype, s, 1, cin), _params(gen, dtype, e, 1, s), _params(gen, dtype, e, 3, s)]
    return {"x": _activations(gen, dtype, (batch, h, w, cin)), "params": [t for p in params for t in p],
            "scratch": torch.empty((batch, h, w, s), dtype=TORCH[dtype], device="cuda"),
            "out": torch.zeros((batch, h, w, 2 * e), dtype=TORCH[dtype], device="cuda")}


def _out_extent(case):
    oh, ow = ((case[d] + 2 * case["pad"] - case["k"]) // case["s"] + 1 for d in ("h", "w"))
    if case["pool"] == "max":
        return (oh - 3) // 2 + 1, (ow - 3) // 2 + 1
    return (1, 1) if case["pool"] == "avg" else (oh, ow)


def _conv_state(case, gen):
    dtype = case["dtype"]
    cin, cout, h, w, k, s, pad, batch = (case[n] for n in ("cin", "cout", "h", "w", "k", "s", "pad", "batch"))
    weights, bias = _params(gen, dtype, cout, k, cin)
    shape = (batch, h, w, cin)
    x = torch.rand(shape, generator=gen, device="cuda").to(TORCH[dtype]) if cin == 3 else _activations(gen, dtype, shape)
    oh, ow = _out_extent(case)
    out_type = torch.float32 if case["pool"] == "avg" else TORCH[dtype]
    nbytes = B.conv_workspace_bytes(cin, cout, h, w, k, s, pad, batch, DTYPE[dtype])
    return {"x": x, "w": weights, "b": bias, "out": torch.zeros((batch, oh, ow, cout), dtype=out_type, device="cuda"),
            "work": torch.empty(nbytes, dtype=torch.uint8, device="cuda") if nbytes else None, "nbytes": nbytes}


def prepare(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    state = {"net": _net_state, "fire": _fire_state, "conv": _conv_state}[case["kind"]](case, gen)
    state["case"] = case
    torch.cuda.synchronize()        # kernels and biases are complete before the first forward (squeezenet_create asks for it)
    return state


# --------------------------------------------------------------------------------------------------------- one pass
def run(state):
    c = state["case"]
    if c["kind"] == "net":
        forward = B.squeezenet_forward_host if c["host"] else B.squeezenet_forward
        forward(state["net"], state["images"], *state["outs"], state["work"], c["batch"])
        return state["outs"]
    if c["kind"] == "fire":
        B.fire_forward(state["x"], *state["params"], state["scratch"], state["out"], c["cin"], c["s"], c["e"], c["e"], c["h"],
                       c["w"], c["batch"], DTYPE[c["dtype"]])
        return state["out"]
    B.conv_forward_ex(state["x"], state["w"], state["b"], state["out"], c["cin"], c["cout"], c["h"], c["w"], c["k"], c["s"],
                      c["pad"], c["batch"], dtype=DTYPE[c["dtype"]], workspace=state["work"], workspace_bytes=state["nbytes"],
                      fuse_maxpool=c["pool"] == "max", fuse_global_avgpool=c["pool"] == "avg")
    return state["out"]


# ---------------------------------------------------------------------------------------------------- what it takes
def work(case):
    """Bytes: operands and results, each once (no intermediate of the network or of a fire layer).  Flops: two per
    product of the convolutions' definition."""
    z, n = SIZE[case["dtype"]], case["batch"]
    if case["kind"] == "net":
        params = sum(cin * cout * k * k for _, cin, cout, k, *_ in synth.SQUEEZENET_CONVS)
        biases = sum(cout for _, _, cout, *_ in synth.SQUEEZENET_CONVS)
        macs = sum(cin * cout * k * k * ((hw + 2 * pad - k) // s + 1) ** 2
                   for _, cin, cout, k, s, pad, hw in synth.SQUEEZENET_CONVS)
        image = 228 * 228 * 4 if case["packed"] else IMG * IMG * 3
        return {"bytes": n * image * z + params * z + biases * 4 + n * 2 * 1000 * 4, "flops": 2 * n * macs}
    if case["kind"] == "fire":
        cin, s, e, px = case["cin"], case["s"], case["e"], case["h"] * case["w"]
        params = cin * s + 10 * s * e
        return {"bytes": n * px * (cin + 2 * e) * z + params * z + (s + 2 * e) * 4, "flops": 2 * n * px * params}
    oh, ow = ((case[d] + 2 * case["pad"] - case["k"]) // case["s"] + 1 for d in ("h", "w"))
    ph, pw = _out_extent(case)
    params = case["cin"] * case["cout"] * case["k"] ** 2
    out_size = 4 if case["pool"] == "avg" else z
    return {"bytes": n * case["h"] * case["w"] * case["cin"] * z + params * z + case["cout"] * 4 + n * ph * pw * case["cout"] * out_size,
            "flops": 2 * n * oh * ow * params}


# About four times what one pass differs from the same path in 64 bits (activations still rounded to the path's storage
# type after each layer): measured over the listed cases and drawn ones.  2-norm: layers 4.3e-7 (reductions up to 512
# long; 1.3e-6 expected at 4608) / 1.7e-3 / 2.1e-4 in f32 / bf16 / f16, network results 2.3e-7 / 5.5e-4 / 1.1e-4.
# Largest difference: layers 3e-6 / 1.3e-2 / 1.9e-3, network results 8.4e-7 / 2.2e-3 / 5.0e-4.
LAYER_TOL = {"f32": (5e-6, 2e-5), "bf16": (7e-3, 5e-2), "f16": (9e-4, 8e-3)}
NET_TOL = {"f32": (1e-6, 4e-6), "bf16": (2.2e-3, 9e-3), "f16": (4.5e-4, 2e-3)}


def tolerance(case):
    rel, largest = (NET_TOL if case["kind"] == "net" else LAYER_TOL)[case["dtype"]]
    return {"rel": rel, "max": largest}
