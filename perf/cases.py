"""Cases that stand for what a program has this library do: fused-tile runs of CNN
front-ends through ``Net`` / ``Plan`` and their run calls.

A case is one plan and one call: the layer stack, the image size, the frames in the call,
the cut and the tile grids (the method's configuration), the data type and the entry point.
Sizes are those of the repository's workloads and tests (the YOLOv2 front-end and trunk
at 96 ... 1216 pixels, the three-layer stack, single layers and blocks of odd sizes).
Images are uniform on [0, 1), weights He-normal, the folded batch-norm's scale uniform
on [0.5, 1.5) and its bias normal with deviation 0.1; in bf16 cases images and weights
are bf16 values, as the library holds them.
"""
import math

import torch

import paper_2107_06960_gb300 as mf

C3, C1, MAX = 3, 1, 0  # a 3x3 or 1x1 convolution, or a 2x2 max-pool


def _c3(f):
    return (C3, f)


def _c1(f):
    return (C1, f)


_POOL = (MAX, 0)
_FRONT = [_c3(32), _POOL, _c3(64), _POOL, _c3(128), _c1(64), _c3(128), _POOL, _c3(256), _c1(128), _c3(256), _POOL,
          _c3(512), _c1(256), _c3(512), _c1(256)]
STACKS = {
    # the first 16 layers of YOLOv2: the network the method is evaluated on
    "front16": _FRONT,
    # the YOLOv2 trunk up to its route layer (weight-heavy layers at 1/32 resolution)
    "trunk25": _FRONT + [_c3(512), _POOL, _c3(1024), _c1(512), _c3(1024), _c1(512), _c3(1024), _c3(1024), _c3(1024)],
    # the smallest stack: two convolutions around a pool
    "tiny3": [_c3(8), _POOL, _c3(16)],
    # bottleneck blocks of the front-end by themselves, for a program that runs single layer
    # groups (no pool, so that any map size goes); the input is a feature map
    "block64": [_c3(128), _c1(64), _c3(128)],
    "block128": [_c3(256), _c1(128), _c3(256)],
    "block256": [_c3(512), _c1(256), _c3(512)],
}
IN_C = {"front16": 3, "trunk25": 3, "tiny3": 3, "block64": 64, "block128": 128, "block256": 256}


def _case(name, stack, h, w, batch, cut, grid1, grid2=(1, 1), dtype="bf16", call="run"):
    return {"name": name, "stack": stack, "h": h, "w": w, "batch": batch, "cut": cut, "n1": grid1[0], "m1": grid1[1],
            "n2": grid2[0], "m2": grid2[1], "dtype": dtype, "call": call}


def listed():
    return [
        # the smallest call: three layers of one 64x64 image; launch and set-up latency
        _case("tiny3_64", "tiny3", 64, 64, 1, 0, (2, 2)),
        # a small image, as cameras of the smallest size give: latency of 13 dependent layers
        _case("front_224", "front16", 224, 224, 1, 8, (2, 2), (1, 1)),
        # the detector's usual input, one layer group (the plan of the 416x416 workload)
        _case("front_416", "front16", 416, 416, 1, 0, (3, 3)),
        # the benchmark: one 608x608 frame, cut after layer 7, 5x5 and 2x2 tiles
        _case("front_608", "front16", 608, 608, 1, 8, (5, 5), (2, 2)),
        # a server's batch of the same frames in one launch
        _case("front_608_b16", "front16", 608, 608, 16, 8, (5, 5), (2, 2)),
        # the largest: eight 1216x1216 frames, 64 and 16 tiles each
        _case("front_1216_b8", "front16", 1216, 1216, 8, 8, (8, 8), (4, 4)),
        # an oblong picture, an early cut and grids that do not divide the maps
        _case("front_720x1280_b2", "front16", 720, 1280, 2, 4, (3, 5), (2, 3)),
        # the longer network, weight-heavy at the end
        _case("trunk_608", "trunk25", 608, 608, 1, 8, (5, 5), (2, 2)),
        # one block of layers on a feature map of odd size, as a layer group run by itself
        _case("block128_75x101_b3", "block128", 75, 101, 3, 0, (2, 3)),
        # one frame from pinned host memory and its result back to it, as a camera loop does
        _case("host_608", "front16", 608, 608, 1, 8, (5, 5), (2, 2), "bf16", "host"),
        # single precision in a loop that may not allocate device memory while it runs
        _case("fp32_noalloc_96_b2", "front16", 96, 96, 2, 8, (2, 2), (2, 2), "fp32", "noalloc"),
        # single precision at the detector's usual input
        _case("fp32_416", "front16", 416, 416, 1, 0, (3, 3), (1, 1), "fp32"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["front", "front", "front", "batch", "trunk", "block", "block", "tiny", "host", "fp32", "noalloc"])
    g = lambda hi: (rng.randint(1, hi), rng.randint(1, hi))
    if kind == "tiny":
        h, w = 2 * _log_int(rng, 8, 128), 2 * _log_int(rng, 8, 128)
        return _draw_case("tiny3", h, w, rng.randint(1, 4), 0, g(3), g(1))
    if kind == "block":
        stack = rng.choice(["block64", "block128", "block256"])
        h, w = _log_int(rng, 7, 152), _log_int(rng, 7, 152)
        return _draw_case(stack, h, w, rng.randint(1, 4), 0, g(3), g(1))
    if kind == "trunk":
        h, w = 32 * _log_int(rng, 3, 19), 32 * _log_int(rng, 3, 19)
        return _draw_case("trunk25", h, w, rng.randint(1, 2), 8, g(5), g(2))
    cut = rng.choice([0, 2, 4, 8, 8, 12])
    if kind == "noalloc":  # what the fixed area holds
        return _draw_case("front16", 16 * rng.randint(2, 6), 16 * rng.randint(2, 6), rng.randint(1, 2), 8, g(3), g(2),
                          "fp32", "noalloc")
    if kind == "fp32":
        return _draw_case("front16", 16 * _log_int(rng, 2, 26), 16 * _log_int(rng, 2, 26), 1, cut, g(4), g(3), "fp32")
    if kind == "batch":
        h, w = 16 * _log_int(rng, 6, 38), 16 * _log_int(rng, 6, 38)
        return _draw_case("front16", h, w, rng.randint(2, 16), cut or 8, g(6), g(3))
    # one or two frames of a camera, up to the largest picture
    h, w = 16 * _log_int(rng, 2, 76), 16 * _log_int(rng, 2, 76)
    if kind == "host":
        return _draw_case("front16", min(h, 608), min(w, 608), 1, cut, g(5), g(3), "bf16", "host")
    return _draw_case("front16", h, w, rng.randint(1, 2), cut, g(6), g(4))


def _draw_case(stack, h, w, batch, cut, g1, g2, dtype="bf16", call="run"):
    c = _case("", stack, h, w, batch, cut, g1, g2, dtype, call)
    del c["name"]
    return c


def _shapes(case):
    """(kind, c_in, c_out, h_in, w_in) of every layer."""
    h, w, c = case["h"], case["w"], IN_C[case["stack"]]
    out = []
    for kind, f in STACKS[case["stack"]]:
        n = c if kind == MAX else f
        out.append((kind, c, n, h, w))
        if kind == MAX:
            h, w = h // 2, w // 2
        c = n
    return out, (h, w, c)


def _data(case, seed):
    """The image batch (NHWC) and every convolution's (weights, scale, bias), on the GPU, in
    fp32; in bf16 cases the image and the weights are bf16 values."""
    gen = torch.Generator(device="cuda").manual_seed(seed * 7919 + 17)
    bf16 = case["dtype"] == "bf16"
    x = torch.rand((case["batch"], case["h"], case["w"], IN_C[case["stack"]]), generator=gen, device="cuda")
    params = []
    for kind, ci, co, _, _ in _shapes(case)[0]:
        if kind == MAX:
            params.append(None)
            continue
        wt = torch.randn((co, ci, kind, kind), generator=gen, device="cuda") * math.sqrt(2.0 / (ci * kind * kind))
        scale = torch.rand((co,), generator=gen, device="cuda") + 0.5
        bias = torch.randn((co,), generator=gen, device="cuda") * 0.1
        params.append((wt.bfloat16().float() if bf16 else wt, scale, bias))
    return (x.bfloat16().float() if bf16 else x), params


def prepare(case, seed):
    x, params = _data(case, seed)
    layers = [("max", 2, 2, 0, 0) if k == MAX else ("conv", k, 1, k // 2, f) for k, f in STACKS[case["stack"]]]
    net = mf.Net(layers, case["h"], case["w"], IN_C[case["stack"]])
    net.set_params([None if p is None else tuple(t.cpu().numpy() for t in p) for p in params])
    grids = [(case["n1"], case["m1"])] + ([(case["n2"], case["m2"])] if case["cut"] else [])
    bf16 = case["dtype"] == "bf16"
    plan = mf.Plan(net, cut=case["cut"] or None, grids=grids, batch=case["batch"], dtype=mf.BF16 if bf16 else mf.FP32)
    x = x.bfloat16() if bf16 else x
    shape = (case["batch"],) + _shapes(case)[1]
    if case["call"] == "host":
        inp, out = x.cpu().pin_memory(), torch.zeros(shape, dtype=x.dtype).pin_memory()
    else:
        inp, out = x.contiguous(), torch.zeros(shape, dtype=x.dtype, device="cuda")
    return {"net": net, "plan": plan, "x": inp, "out": out, "call": case["call"]}


def run(state):
    plan, x, out = state["plan"], state["x"], state["out"]
    if state["call"] == "host":
        plan.run_host(x, out)
    elif state["call"] == "noalloc":
        plan.run_noalloc(x, out)
    else:
        plan.run(x, out)
    return out


def work(case):
    """One pass over the unfused network: the image, the weights, scales and biases read once,
    the output written once; two operations a multiply-add."""
    size = 2 if case["dtype"] == "bf16" else 4
    shapes, (ho, wo, co) = _shapes(case)
    b = case["batch"]
    bytes_ = size * b * (case["h"] * case["w"] * IN_C[case["stack"]] + ho * wo * co)
    flops = 0
    for kind, ci, cn, h, w in shapes:
        if kind != MAX:
            flops += 2 * b * h * w * ci * cn * kind * kind
            bytes_ += size * ci * cn * kind * kind + 8 * cn
    return {"bytes": bytes_, "flops": flops}


def tolerance(case):
    """About four times what a correct run shows against exact()."""
    if case["dtype"] == "fp32":  # fp32 sums of up to 4608 products in each of 13 layers: 2e-6 seen
        return {"rel": 1e-5, "max": 1e-4}
    # every layer's output is rounded to bf16 (2^-9 relative): 2.2e-3 seen after two layers, 2.9e-3
    # after three, 6.7e-3 after 13, 8.3e-3 after 22
    rel = {"front16": 2.5e-2, "trunk25": 3.5e-2}.get(case["stack"], 1.2e-2)
    return {"rel": rel, "max": 8 * rel}


def exact(case, seed):
    """The stack layer by layer in fp64: a convolution as one matrix product per tap."""
    x, params = _data(case, seed)
    outs = []
    for f in range(case["batch"]):
        a = x[f].double()
        for (kind, ci, co, h, w), prm in zip(_shapes(case)[0], params):
            if kind == MAX:
                a = a.reshape(h // 2, 2, w // 2, 2, ci).amax(dim=(1, 3))
                continue
            wt, scale, bias = (t.double() for t in prm)
            p = kind // 2
            pad = torch.nn.functional.pad(a, (0, 0, p, p, p, p))
            z = torch.zeros((h * w, co), dtype=torch.float64, device=a.device)
            for ky in range(kind):
                for kx in range(kind):
                    z.addmm_(pad[ky:ky + h, kx:kx + w].reshape(h * w, ci), wt[:, :, ky, kx].t())
            z = z * scale + bias
            a = torch.where(z > 0, z, 0.1 * z).reshape(h, w, co)
        outs.append(a)
    return torch.stack(outs)
