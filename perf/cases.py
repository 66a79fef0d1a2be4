"""Workloads this library is timed on, through its public entry points.

Every case is one thing a user has the library do: a single pruned layer on NHWC tensors
(cadnn_conv2d, cadnn_fc), or the forward pass of a whole pruned network (PackedModel.forward /
forward_host, i.e. cadnn_forward / cadnn_forward_host) built the default way.  Layer shapes,
networks, densities and batch sizes are those of the repository's workloads (workloads/models.py):
the single 3x3 layer, ResNet-50, int8 VGG-16, MobileNet-V2, the batch x density sweep of ResNet-50,
Inception-V3 and int8 ResNet-50.  Weights, masks and inputs are drawn from the seed, with the
distributions of workloads/gen.py.

  listed()              the fixed cases
  draw(rng)             one more case of the same ranges
  prepare(case, seed)   inputs and packed weights / network, on the GPU
  run(state)            one pass; returns the outputs
  work(case)            bytes and operations one pass cannot do without
  tolerance(case)       agreement to expect of another correct implementation
"""
import functools
import math

import numpy as np
import torch

from paper_1905_00571_b200 import binding
from paper_1905_00571_b200.network import PackedModel
from workloads import gen, models

# network -> (default image, conv density, fc density) of the repository's configurations
NETS = {"resnet50": (224, 0.125, 0.10), "mobilenet_v2": (224, 0.25, 0.25), "inception_v3": (299, 0.125, 0.10),
        "vgg16": (224, 0.08, 0.04), "resnet50_int8": (224, 0.125, 0.10)}


def _net(name, net, batch, image=None, density=None, host=False):
    im, d, fd = NETS[net]
    return {"name": name, "kind": "net", "net": net, "batch": batch, "image": image or im, "density": density or d,
            "fc_density": fd, "host": host}


def _conv(name, dtype, batch, c_in, c_out, k, stride, pad, h, w, density, residual=False):
    return {"name": name, "kind": "conv", "dtype": dtype, "batch": batch, "c_in": c_in, "c_out": c_out, "k": k, "stride": stride,
            "pad": pad, "h": h, "w": w, "density": density, "residual": residual}


def _fc(name, dtype, batch, c_in, c_out, density):
    return {"name": name, "kind": "fc", "dtype": dtype, "batch": batch, "c_in": c_in, "c_out": c_out, "density": density}


def listed():
    return [
        # the classifier of the pruned ResNet-50 on one image: the smallest call, all latency
        _fc("fc_f32_b1", "f32", 1, 2048, 1000, 0.10),
        # the second FC layer of VGG-16 on a serving batch, int8
        _fc("fc_s8_b32", "s8", 32, 4096, 4096, 0.04),
        # the single-layer configuration: 64 -> 64 3x3 on a 56x56 map, 10 % of the weights, one image
        _conv("conv_f32_b1", "f32", 1, 64, 64, 3, 1, 1, 56, 56, 0.10),
        # an unpadded layer of odd size (the 80 -> 192 3x3 layer of Inception-V3) on a few images
        _conv("conv_f32_ragged", "f32", 5, 80, 192, 3, 1, 0, 73, 73, 0.125),
        # the headline: pruned ResNet-50, single-image latency, on device tensors ...
        _net("resnet50_f32_b1", "resnet50", 1),
        # ... and from pinned host memory to host memory
        _net("resnet50_f32_b1_host", "resnet50", 1, host=True),
        # a small batch of a less pruned ResNet-50
        _net("resnet50_f32_b8_d25", "resnet50", 8, density=0.25),
        # offline throughput: the largest batch of the sweep
        _net("resnet50_f32_b128", "resnet50", 128),
        # single-image latency of the network with depthwise layers and ReLU6
        _net("mobilenet_v2_f32_b1", "mobilenet_v2", 1),
        # int8 VGG-16, single image
        _net("vgg16_s8_b1", "vgg16", 1),
        # int8 ResNet-50 (int8 residuals, strided layers), a serving batch
        _net("resnet50_s8_b8", "resnet50_int8", 8),
        # Inception-V3, single image: rectangular kernels, concatenations, average pools
        _net("inception_v3_f32_b1", "inception_v3", 1),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(_log(rng, lo, hi)))))


def draw(rng):
    kind = rng.choice(["net", "net", "conv", "fc"])
    if kind == "fc":
        c = _fc("", rng.choice(["f32", "s8"]), _log_int(rng, 1, 64), _log_int(rng, 256, 25088), _log_int(rng, 100, 4096),
                round(_log(rng, 0.03, 0.3), 4))
    elif kind == "conv":
        k = rng.choice([1, 1, 3, 3, 5])
        dtype = rng.choice(["f32", "f32", "s8"])
        c = _conv("", dtype, _log_int(rng, 1, 32), _log_int(rng, 16, 512), _log_int(rng, 16, 512), k, rng.choice([1, 1, 2]),
                  rng.choice([k // 2, k // 2, 0]), _log_int(rng, 7, 112), _log_int(rng, 7, 112), round(_log(rng, 0.05, 0.5), 4),
                  residual=rng.choice([False, True]))
    else:
        net = rng.choice(sorted(NETS))
        im, d, _ = NETS[net]
        c = _net("", net, _log_int(rng, 1, 32), image=rng.randint(im - 64, im + 32), density=round(d * _log(rng, 0.5, 4.0), 4),
                 host=rng.random() < 0.2)
    del c["name"]
    most = 0.9 * work(_largest())["flops"]
    while work(c)["flops"] > most or (c["kind"] == "conv" and 4 * c["batch"] * c["h"] * c["w"] * (c["c_in"] + c["c_out"]) > 2e9):
        c["batch"] = max(1, c["batch"] // 2)
        c["density"] = round(c["density"] / 1.5, 4)
    return c


@functools.lru_cache(maxsize=1)
def _largest():
    return max(listed(), key=lambda c: work(c)["flops"])


@functools.lru_cache(maxsize=8)
def _skeleton(net, image):
    """The network's layer list with every weight kept, as (model, layer shapes); its weights are not used."""
    narrow = 64   # VGG-16's FC layers hold nearly all of its weights: generated narrow, then widened to 4096
    dense = {"mobilenet_v2": {}, "vgg16": {"fc_density": 1.0, "fc_width": narrow}}.get(net, {"fc_density": 1.0})
    m = getattr(models, net)(image=image, density=1.0, **dense)
    shapes = []
    for op in m.ops:
        shape = None if op.w is None else op.w.shape
        if net == "vgg16" and op.kind == "fc":
            c_in, c_out = (4096 if c == narrow else c for c in (op.c_in, op.c_out))
            op.scale = np.resize(op.scale, c_out) * np.float32(math.sqrt(op.c_in / c_in))
            op.bias = np.resize(op.bias, c_out)
            op.c_in, op.c_out, shape = c_in, c_out, (c_out, 1, 1, c_in)
        shapes.append(None if op.w is None else (shape, op.w.dtype))
        op.w = None
    return m, shapes


def _density(case, op):
    """Depthwise layers and the first conv of the float networks and of int8 ResNet-50 stay dense."""
    if op.kind == "fc":
        return case["fc_density"]
    if op.groups > 1 or (op.c_in <= 4 and case["net"] != "vgg16"):
        return 1.0
    return min(1.0, case["density"])


def _mask(score, density):
    """uint8 mask of the round(density * size) largest scores."""
    flat = torch.zeros(score.numel(), dtype=torch.uint8, device=score.device)
    flat[torch.topk(score.reshape(-1), gen.keep_count(density, score.numel()), sorted=False).indices] = 1
    return flat.reshape(score.shape)


def _weights(g, shape, dtype, density):
    """Weights and mask of one layer: float N(0, 2 / fan_in) pruned by magnitude, or int8 codes pruned at random."""
    w = torch.randn(shape, generator=g, device="cuda")
    if dtype == np.int8:
        w = (w * 40.0).round_().clamp_(-127, 127).to(torch.int8)
        score = torch.rand(shape, generator=g, device="cuda") if density < 1.0 else None
    else:
        w *= math.sqrt(2.0 / float(np.prod(shape[1:])))
        score = w.abs() if density < 1.0 else None
    mask = None if score is None else _mask(score, density)
    kept = 1.0
    if mask is not None:
        kept = float((w.double() ** 2 * mask).sum() / (w.double() ** 2).sum()) if dtype != np.int8 else density
    return w.cpu().numpy(), None if mask is None else mask.cpu().numpy(), kept


def _codes(g, shape):
    return (torch.randn(shape, generator=g, device="cuda") * (127.0 / 3.0)).round_().clamp_(-127, 127)


def prepare(case, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return _prepare_net(case, g) if case["kind"] == "net" else _prepare_layer(case, g)


def _prepare_net(case, g):
    base, shapes = _skeleton(case["net"], case["image"])
    m = models.Model(base.name, base.dtype, base.in_shape, seed=base.seed, n_slots=base.n_slots)
    for op, shape in zip(base.ops, shapes):
        op = models.Op(**vars(op))
        if shape is not None:
            op.density = _density(case, op)
            op.w, op.mask, kept = _weights(g, shape[0], shape[1], op.density)
            op.scale = (op.scale / math.sqrt(kept)).astype(np.float32)   # keeps the activations' range, as the workloads do
        m.ops.append(op)
    pm = PackedModel(m, case["batch"])
    for op in m.ops:
        op.w = op.mask = None    # a deployed program keeps the packed form only
    h, w, c = m.in_shape
    shape = (case["batch"], h, w, c)
    x = _codes(g, shape).to(torch.int8) if m.dtype == "s8" else torch.randn(shape, generator=g, device="cuda")
    y = pm.new_output()
    if case["host"]:
        x = x.cpu().pin_memory()
        y = torch.empty(pm.out_shape, dtype=pm.out_dtype).pin_memory()
    return {"case": case, "pm": pm, "x": x, "y": y}


def _prepare_layer(case, g):
    s8 = case["dtype"] == "s8"
    k = case.get("k", 1)
    w, mask, kept = _weights(g, (case["c_out"], k, k, case["c_in"]), np.int8 if s8 else np.float32, case["density"])
    if case["kind"] == "fc":
        d = binding.make_desc(case["c_in"], case["c_out"], batch_hint=case["batch"], dtype=case["dtype"])
        xs, ys = (case["batch"], case["c_in"]), (case["batch"], case["c_out"])
    else:
        d = binding.make_desc(case["c_in"], case["c_out"], k, k, case["stride"], case["pad"], 1, case["h"], case["w"], case["batch"],
                              case["dtype"])
        xs, ys = (case["batch"], case["h"], case["w"], case["c_in"]), (case["batch"],) + _out_hw(case) + (case["c_out"],)
    x = torch.randn(xs, generator=g, device="cuda").relu_()       # a feature map as a ReLU layer leaves it
    scale = torch.rand(case["c_out"], generator=g, device="cuda") + 0.5
    bias = torch.randn(case["c_out"], generator=g, device="cuda") * 0.1
    residual = torch.randn(ys, generator=g, device="cuda").relu_() if case.get("residual") else None
    if s8:
        x = (x * (127.0 / 3.0)).round_().clamp_(0, 127).to(torch.int8)
        # requantize the sums of c_in k k density products of codes (rms 40 and 30) to an rms of a third of the range
        scale *= (127.0 / 3.0) / (40.0 * 30.0 * math.sqrt(case["c_in"] * k * k * case["density"]))
        bias *= 127.0 / 3.0
        if residual is not None:
            residual = (residual * (127.0 / 3.0)).round_().clamp_(0, 127).to(torch.int8)
    packed = binding.cadnn_pack_q8(d, w, mask) if s8 else binding.cadnn_pack(d, w, mask)
    y = torch.empty(ys, dtype=torch.int8 if s8 else torch.float32, device="cuda")
    return {"case": case, "w": packed, "x": x, "y": y, "scale": scale, "bias": bias, "residual": residual}


def run(s):
    c = s["case"]
    if c["kind"] == "net":
        return s["pm"].forward_host(s["x"], s["y"]) if c["host"] else s["pm"].forward(s["x"], s["y"])
    if c["kind"] == "fc":
        return binding.cadnn_fc(s["w"], s["x"], s["y"], scale=s["scale"], bias=s["bias"], act="relu")
    return binding.cadnn_conv2d(s["w"], s["x"], s["y"], scale=s["scale"], bias=s["bias"], residual=s["residual"], act="relu",
                                residual_scale=0.5)


def _out_hw(case):
    k, s, p = case["k"], case["stride"], case["pad"]
    return (case["h"] + 2 * p - k) // s + 1, (case["w"] + 2 * p - k) // s + 1


def work(case):
    """Input and output once, the compressed weights once (a value and a 16-bit position per kept weight; dense layers
    the value alone), two operations per kept weight and output position.  What passes between the layers of a network
    is not counted: nothing but the present split into layers makes it travel."""
    flops = nbytes = 0.0
    if case["kind"] == "net":
        m, shapes = _skeleton(case["net"], case["image"])
        for op, shape in zip(m.ops, shapes):
            if shape is not None:
                d, n, e = _density(case, op), float(np.prod(shape[0])), np.dtype(shape[1]).itemsize
                nbytes += d * n * (e + (2 if d < 1.0 else 0)) + 8 * op.c_out
                flops += 2 * d * n * op.out_hw[0] * op.out_hw[1] * case["batch"]
        e = 1 if m.dtype == "s8" else 4
        last = m.ops[-1]
        nbytes += case["batch"] * (e * float(np.prod(m.in_shape)) + 4 * last.c_out)
    else:
        k, e = case.get("k", 1), 1 if case["dtype"] == "s8" else 4
        nnz = case["density"] * case["c_in"] * case["c_out"] * k * k
        px_in, px_out = (1, 1) if case["kind"] == "fc" else (case["h"] * case["w"], int(np.prod(_out_hw(case))))
        flops = 2 * nnz * px_out * case["batch"]
        nbytes = nnz * (e + 2) + 8 * case["c_out"] + e * case["batch"] * (px_in * case["c_in"]
                                                                          + px_out * case["c_out"] * (2 if case.get("residual") else 1))
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    """int8 results are exact; float32 sums in any order agree to about 1e-5, a chain of fifty to a hundred such layers to 3e-5."""
    if case["kind"] == "net":
        if case["net"] == "vgg16":
            return "exact"
        return {"rel": 1e-5} if case["net"] == "resnet50_int8" else {"rel": 3e-5}
    return "exact" if case["dtype"] == "s8" else {"rel": 1e-5}
