"""The workloads whose speed this library is judged by, through its public entry points.

A case is a dict of plain values.  "op" names the entry point:
  conv     Plan.conv2d on device tensors, half or fp32 mode (3 x 3, or 5 x 5 with "r": 5)
  int8     Plan.conv2d_int8 with the input scale derived from the data
  filter   Plan.filter_transform, what loading a layer's weights costs
  host     Plan.conv2d_host, page-locked host tensors in and out
  stack    the 13 convolution layers of the VGG-16 configuration with their five fused max-pools
Activations are ReLU'd standard normals and weights are He-normal, as in synth/inputs.py, drawn on the
GPU from the seed.  Plans, transformed filters, outputs and workspaces are what a program keeps between
calls, so `prepare` makes them; a pass is the call alone.
"""
import math

import torch

import paper_2512_18453_b200 as nv
from synth import VGG16_LAYERS, point_set


def _conv(name, m, points, N, H, W, C, K, op="conv", mode="fp16", r=3, relu=True):
    return {"name": name, "op": op, "mode": mode, "m": m, "r": r, "points": points,
            "N": N, "H": H, "W": W, "C": C, "K": K, "relu": relu}


def listed():
    return [
        # the smallest call: one 16 x 16 image, 8 -> 8 channels, fp32 mode; latency and launches only
        _conv("f2_fp32_16x16_c8", 2, "std", 1, 16, 16, 8, 8, mode="fp32", relu=False),
        # the fp32 mode as an accuracy reference of a real layer: a batch of 8, 56 x 56, 64 channels
        _conv("f4_fp32_56x56_c64", 4, "std", 8, 56, 56, 64, 64, mode="fp32"),
        # the same layer in half precision with the discovered points: a small ordinary call
        _conv("f4_56x56_c64", 4, "nova", 8, 56, 56, 64, 64),
        # the VGG conv3-shaped layer at batch 32, the library's headline workload
        _conv("f6_56x56_c256", 6, "nova", 32, 56, 56, 256, 256, relu=False),
        # the VGG conv4-shaped layer at batch 32 with the largest tile
        _conv("f8_28x28_c512", 8, "nova", 32, 28, 28, 512, 512),
        # nothing divides anything: ragged image, channels not a multiple of 64, a point set that is
        # not symmetric about 0 (dense transforms)
        _conv("f6_45x61_c200_k328", 6, "asym", 7, 45, 61, 200, 328),
        # a 5 x 5 filter
        _conv("f4r5_56x56_c128", 4, "nova", 8, 56, 56, 128, 128, r=5),
        # the INT8 pipeline at the tile size where its error is usable, scale of the input from the data
        _conv("f4_int8_56x56_c256", 4, "dyadic", 32, 56, 56, 256, 256, op="int8"),
        # a layer's weights made ready when a model is loaded
        {"name": "filter_f6_c512", "op": "filter", "mode": "fp16", "m": 6, "r": 3, "points": "nova", "C": 512, "K": 512},
        # host tensors in and out
        _conv("host_f6_56x56_c256", 6, "nova", 8, 56, 56, 256, 256, op="host"),
        # a whole network for one image: thirteen small dependent calls, what serving one request costs
        {"name": "vgg16_batch1", "op": "stack", "mode": "fp16", "m": 4, "r": 3, "points": "dyadic", "N": 1, "HW": 224},
        # the same network at batch 32, the largest workload (F(6,3): with F(8,3) on half storage the
        # thirteen layers' rounding errors of some 40 % each make two correct runs differ by 20 %)
        {"name": "vgg16_batch32", "op": "stack", "mode": "fp16", "m": 6, "r": 3, "points": "half", "N": 32, "HW": 224},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _channels(rng, lo, hi, step):
    """Half the time a power of two times `step`'s range, otherwise any multiple of `step`."""
    c = _log_int(rng, lo, hi)
    if rng.random() < 0.5:
        c = 1 << int(round(math.log2(c)))
    return max(lo, min(hi, (c + step - 1) // step * step))


def draw(rng):
    op = rng.choices(["conv", "conv_r5", "conv_fp32", "int8", "filter", "host", "stack"], [8, 2, 3, 3, 2, 1, 2])[0]
    if op == "stack":
        m, points = rng.choice([(4, "dyadic"), (6, "half")])
        return {"op": "stack", "mode": "fp16", "m": m, "r": 3, "points": points, "N": _log_int(rng, 1, 16),
                "HW": 32 * rng.randint(2, 7)}
    r = 5 if op == "conv_r5" else 3
    m = rng.choice([2, 4, 6] if r == 5 else [2, 4, 6] if op in ("conv_fp32", "host") else [4] if op == "int8" else [2, 4, 6, 8])
    kinds = {2: ["std", "asym"], 4: ["std", "nova", "dyadic", "asym"], 6: ["half", "nova", "asym"], 8: ["nova"]}
    points = rng.choice(["dyadic", "nova"]) if op == "int8" else rng.choice(kinds[m + r - 3])
    mode = "fp32" if op == "conv_fp32" else "fp16"
    step = 16 if op == "int8" else 8
    C, K = _channels(rng, step, 512, step), _channels(rng, step, 512, step)
    if op == "filter":
        return {"op": "filter", "mode": mode, "m": m, "r": r, "points": points, "C": max(C, 64), "K": max(K, 64)}
    H = _log_int(rng, 7, 112)
    W = H if rng.random() < 0.5 else _log_int(rng, 7, 112)
    N = _log_int(rng, 1, 32)
    # no more than the batch of the headline layer (the fp32 mode: than its listed layer), in multiplications
    most = {"fp32": 8 * 56 * 56 * 64 * 64, "fp16": 32 * 56 * 56 * 256 * 256}[mode] // (4 if op == "host" else 1)
    most = most * 9 // (r * r)
    while N * H * W * C * K > most:
        if N > 1:
            N //= 2
        elif C >= K and C > step:
            C = max(step, C // 2 // step * step)
        else:
            K = max(step, K // 2 // step * step)
    c = _conv("", m, points, N, H, W, C, K, op="conv" if op.startswith("conv") else op, mode=mode, r=r, relu=rng.random() < 0.7)
    del c["name"]
    return c


# ---------------------------------------------------------------------------- inputs
def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _normal(g, *shape):
    return torch.randn(*shape, generator=g, device="cuda", dtype=torch.float32)


def _points(case):
    return point_set(case["points"], case["m"] + case["r"] - 3)


def _layers(case):
    """(H, C, K, flags) of the 13 layers of a stack."""
    h, out = case["HW"], []
    for ci, co, pool in VGG16_LAYERS:
        out.append((h, max(ci, 8), co, nv.RELU | (nv.POOL2X2 if pool else 0)))
        h = h // 2 if pool else h
    return out


def prepare(case, seed):
    g = _gen(seed)
    mode = nv.FP32 if case["mode"] == "fp32" else nv.FP16_F32ACC
    dtype = torch.float32 if mode == nv.FP32 else torch.float16
    plan = nv.Plan(case["m"], _points(case), mode, r=case["r"])
    s = {"op": case["op"], "plan": plan}
    r = case["r"]
    if case["op"] == "stack":
        N = case["N"]
        x = _normal(g, N, case["HW"], case["HW"], 8).relu_()
        x[..., 3:] = 0                                  # three colour channels, padded to 8
        s["x"], s["layers"], ws = x.to(dtype), [], 256
        for i, (h, C, K, flags) in enumerate(_layers(case)):
            w = _normal(g, K, 3, 3, C) * math.sqrt(2.0 / (9 * (3 if i == 0 else C)))
            if i == 0:
                w[..., 3:] = 0
            ho = h // 2 if flags & nv.POOL2X2 else h
            y = torch.empty(N, ho, ho, K, dtype=dtype, device="cuda")
            s["layers"].append((plan.filter_transform(w.to(dtype)), y, flags))
            ws = max(ws, plan.workspace_bytes(N, h, h, C, K))
        s["ws"] = torch.empty(ws, dtype=torch.uint8, device="cuda")
        return s
    C, K = case["C"], case["K"]
    w = (_normal(g, K, r, r, C) * math.sqrt(2.0 / (r * r * C))).to(dtype)
    if case["op"] == "filter":
        s["w"] = w
        return s
    N, H, W = case["N"], case["H"], case["W"]
    s["flags"] = nv.RELU if case["relu"] else 0
    x = _normal(g, N, H, W, C).relu_().to(dtype)
    y = torch.empty(N, H, W, K, dtype=dtype, device="cuda")
    if case["op"] == "int8":
        s["U"], s["scale"] = plan.filter_transform_int8(w, nv.QUANT_PER_CHANNEL)
        ws = plan.int8_workspace_bytes(N, H, W, C, K)
    else:
        s["U"] = plan.filter_transform(w)
        ws = plan.workspace_bytes(N, H, W, C, K)
    s["ws"] = torch.empty(ws, dtype=torch.uint8, device="cuda")
    if case["op"] == "host":
        s["x"] = x.cpu().pin_memory()
        s["y"] = torch.empty(N, H, W, K, dtype=dtype, pin_memory=True)
        s["x_stage"], s["y_stage"] = torch.empty_like(x), y
    else:
        s["x"], s["y"] = x, y
    return s


def run(s):
    op, plan = s["op"], s["plan"]
    if op == "conv":
        return plan.conv2d(s["x"], s["U"], s["y"], s["ws"], s["flags"])
    if op == "int8":
        return plan.conv2d_int8(s["x"], s["U"], s["scale"], 0.0, s["y"], s["ws"], s["flags"])
    if op == "filter":
        return plan.filter_transform(s["w"])
    if op == "host":
        return plan.conv2d_host(s["x"], s["U"], s["y"], s["x_stage"], s["y_stage"], s["ws"], s["flags"])
    a, features = s["x"], []                            # the feature maps of every layer, as a detector takes them
    for U, y, flags in s["layers"]:
        a = plan.conv2d(a, U, y, s["ws"], flags)
        features.append(a)
    return features


# ---------------------------------------------------------------------------- work and tolerance
def _conv_work(case, N, H, W, C, K):
    """Floating-point operations of the transformed-domain product, and the bytes of U."""
    n = case["m"] + case["r"] - 1
    tiles = N * -(-H // case["m"]) * -(-W // case["m"])
    elt = 1 if case["op"] == "int8" else 4 if case["mode"] == "fp32" else 2
    return 2.0 * n * n * tiles * C * K, n * n * C * K * elt


def work(case):
    elt = 4 if case["mode"] == "fp32" else 2
    if case["op"] == "stack":
        flops, nbytes = 0, elt * case["N"] * case["HW"] ** 2 * 8
        for h, C, K, flags in _layers(case):
            f, b = _conv_work(case, case["N"], h, h, C, K)
            ho = h // 2 if flags & nv.POOL2X2 else h
            flops, nbytes = flops + f, nbytes + b + elt * case["N"] * ho * ho * K
        return {"flops": flops, "bytes": nbytes}
    C, K, r = case["C"], case["K"], case["r"]
    if case["op"] == "filter":
        n = case["m"] + r - 1
        return {"flops": 2.0 * K * C * (n * r * r + n * n * r), "bytes": elt * C * K * (r * r + n * n)}
    flops, u = _conv_work(case, case["N"], case["H"], case["W"], C, K)
    return {"flops": flops, "bytes": u + elt * case["N"] * case["H"] * case["W"] * (C + K)}


def tolerance(case):
    """About four times what the present kernels differ by from the same sums in another order (the
    CUDA-core transforms and product; fp32 mode and filters: from float64), over these ranges.  It grows
    with the number of points n = m + r - 1, because the transforms amplify the storage roundings of U and
    V.  Seen: half rel 3.5e-5, 1.2e-4, 1.4e-3, 1.7e-2 for n = 4, 6, 8, 10, largest single difference 0.001,
    0.004, 0.036, 0.6 of the larger of value and root mean square; fp32 7e-8, 4e-7, 4e-6 for n = 4, 6, 8;
    INT8 (codes next to a rounding boundary) 1e-3, 0.04; filter 4e-6, 0.001; stack 1.9e-3 and 4.9e-3 for m = 4, 6."""
    if case["op"] == "stack":
        return {"rel": {4: 8e-3, 6: 2e-2}[case["m"]], "max": 0.12}
    if case["op"] == "filter":
        return {"rel": 1.5e-5, "max": 0.004}
    if case["op"] == "int8":
        return {"rel": 4e-3, "max": 0.16}
    n = case["m"] + case["r"] - 1
    if case["mode"] == "fp32":
        return {"rel": {4: 4e-7, 6: 2e-6, 8: 1.6e-5}[n]}
    return {"rel": {4: 1.5e-4, 6: 5e-4, 8: 6e-3, 10: 3e-2}[n], "max": {4: 0.004, 6: 0.016, 8: 0.15, 10: 0.99}[n]}
