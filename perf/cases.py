"""Performance cases: what a program that serves pruned networks asks of this library.

Three kinds of layer, each called as such a program calls it: packed and planned once, then
enqueued on device tensors over and over.

  conv  pattern-pruned 3x3 convolution (`Packed.plan`, then `run`, or `run_fused` where a
        residual, a pool or a re-quantisation follows the layer)
  gemm  block-pruned matrix product: a 1x1 convolution over pixels, or a fully connected layer
        over rows (`BlockGemm.run`)
  dw    depthwise pattern-pruned 3x3 convolution (`Depthwise.run`)
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2206_10620_b200 import binding, workloads as wl

_T = {"f32": torch.float32, "f16": torch.float16}


# --- cases -------------------------------------------------------------------
def _conv(name, n, hw, c_in, c_out, dtype, prune, *, stride=1, lib=8, relu=True, residual=False, pool=0,
          requant=False):
    h, w = hw
    return {"name": name, "kind": "conv", "n": n, "h": h, "w": w, "c_in": c_in, "c_out": c_out, "stride": stride,
            "dtype": dtype, "prune": prune, "lib": lib, "relu": relu, "residual": residual, "pool": pool,
            "requant": requant}


def _gemm(name, m, k, c_out, dtype, row_keep, col_keep, *, br=32, bc=32, relu=True):
    return {"name": name, "kind": "gemm", "m": m, "k": k, "c_out": c_out, "br": br, "bc": bc,
            "row_keep": row_keep, "col_keep": col_keep, "dtype": dtype, "relu": relu}


def _dw(name, n, hw, c, dtype, *, stride=1, prune=0.0, lib=8, relu=True):
    h, w = hw
    return {"name": name, "kind": "dw", "n": n, "h": h, "w": w, "c": c, "stride": stride, "dtype": dtype,
            "prune": prune, "lib": lib, "relu": relu}


def listed():
    return [
        # the `single` configuration: the smallest call, where the launch and the host path count
        _conv("conv_single_f32", 1, (32, 32), 16, 32, "f32", 0.5),
        # one image at a time (interactive use), fp32, the VGG-16 stack of the benchmark:
        # its first layer (three channels, large image, nothing pruned) ...
        _conv("conv_first_f32_b1", 1, (224, 224), 3, 64, "f32", 0.0),
        # ... a middle layer ...
        _conv("conv_mid_f32_b1", 1, (56, 56), 256, 256, "f32", 0.7),
        # ... and a late one: few pixels, many channels
        _conv("conv_late_f32_b1", 1, (14, 14), 512, 512, "f32", 0.7),
        # a batch through a stage's last layer, with the pool behind it
        _conv("conv_pool_f32_b8", 8, (112, 112), 128, 128, "f32", 0.7, pool=2),
        # ResNet-50's strided layer at the configuration's batch, fp16
        _conv("conv_strided_f16_b32", 32, (56, 56), 128, 128, "f16", 0.6, stride=2),
        # the sweep's largest batch, fp16: offline throughput, the largest call
        _conv("conv_sweep_f16_b256", 256, (28, 28), 256, 256, "f16", 0.5),
        # ResNet-18 in int8 at the configuration's batch: shortcut, ReLU and re-quantisation fused
        _conv("conv_residual_i8_b64", 64, (28, 28), 128, 128, "i8", 0.5, residual=True, requant=True),
        # nothing divides anything: channel counts after structured pruning, a cropped image
        _conv("conv_ragged_f16_b3", 3, (45, 77), 67, 93, "f16", 0.75, lib=12),
        # a 1x1 convolution of ResNet-50 in matrix form, batch 32
        _gemm("gemm_pointwise_f16", 32 * 56 * 56, 256, 128, "f16", 0.4, 0.4),
        # a fully connected layer over a small batch of rows, fp32, no round sizes
        _gemm("gemm_fc_f32", 96, 1000, 1000, "f32", 0.5, 0.5),
        # a MobileNet-shaped depthwise layer, batch 32
        _dw("dw_f16_b32", 32, (56, 56), 128, "f16"),
    ]


# A drawn case moves and computes no more than the largest listed one.
_MOST_BYTES = 200e6
_MOST_KERNEL_PIXELS = 256 * 28 * 28 * 256 * 256 * 0.5     # (filter, channel, output pixel) triples of a convolution
_MOST_GEMM = 2.5e10                                       # entries of x times output channels, dense
_MOST_GEMM_KEPT = 5e9


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _channels(rng, lo, hi):
    """Mostly round channel counts, as networks have; one in three is whatever pruning left."""
    c = _log(rng, lo, hi)
    return c if rng.random() < 1 / 3 else max(16, (c + 8) // 16 * 16)


def draw(rng):
    while True:
        u = rng.random()
        if u < 0.6:
            stride = 2 if rng.random() < 0.25 else 1
            h = _log(rng, 7, 224)
            w = h if rng.random() < 0.6 else _log(rng, 7, 224)
            dtype = rng.choice(["f32", "f16", "i8"])
            c = _conv("", _log(rng, 1, 256), (h, w), _channels(rng, 3, 512), _channels(rng, 16, 512), dtype,
                      round(rng.uniform(0.0, 0.9), 3), stride=stride, lib=rng.choice([4, 8, 12]),
                      relu=rng.random() < 0.8, residual=rng.random() < 0.25,
                      pool=2 if rng.random() < 0.2 else 0, requant=dtype == "i8" and rng.random() < 0.5)
            ho, wo = _out(c)
            if c["pool"] and (ho % 2 or wo % 2):
                c["pool"] = 0
            if c["n"] * ho * wo * c["c_in"] * c["c_out"] > _MOST_KERNEL_PIXELS:
                continue
        elif u < 0.8:
            dtype = rng.choice(["f32", "f16"])
            b = rng.choice([16, 32, 64])
            c = _gemm("", _log(rng, 1, 400000), _channels(rng, 32, 2048), _channels(rng, 32, 2048), dtype,
                      round(rng.uniform(0.2, 1.0), 2), round(rng.uniform(0.2, 1.0), 2), br=b, bc=b,
                      relu=rng.random() < 0.7)
            if c["m"] * c["k"] * c["c_out"] > _MOST_GEMM or c["m"] * _kept(c) > _MOST_GEMM_KEPT:
                continue
        else:
            h = _log(rng, 7, 224)
            c = _dw("", _log(rng, 1, 256), (h, h if rng.random() < 0.6 else _log(rng, 7, 224)),
                    _channels(rng, 16, 1024), rng.choice(["f32", "f16"]), stride=rng.choice([1, 1, 2]),
                    prune=rng.choice([0.0, 0.0, 0.25]), lib=rng.choice([4, 8, 12]), relu=rng.random() < 0.8)
        if work(c)["bytes"] <= _MOST_BYTES:
            del c["name"]
            return c


# --- sizes -------------------------------------------------------------------
def _out(c):
    s = c["stride"]
    return (c["h"] - 1) // s + 1, (c["w"] - 1) // s + 1


def _survivors(c):
    k = c["c_in"] * c["c_out"]
    return k - int(round(c["prune"] * k))


def _edge_blocks(extent, block):
    """(size, how many) of the pruning blocks along one side of the matrix."""
    full, rest = divmod(extent, block)
    return [(block, full)] * (full > 0) + [(rest, 1)] * (rest > 0)


def _kept(c):
    return sum(nr * nc * int(round(c["row_keep"] * r)) * int(round(c["col_keep"] * k))
               for r, nr in _edge_blocks(c["c_out"], c["br"]) for k, nc in _edge_blocks(c["k"], c["bc"]))


def work(case):
    """Input and result once, the kept weights with two index bytes a kernel (none in the block-pruned
    form), the bias; two operations per kept weight and output element."""
    c = case
    if c["kind"] == "gemm":
        b = 4 if c["dtype"] == "f32" else 2
        kept = _kept(c)
        return {"bytes": c["m"] * (c["k"] + c["c_out"]) * b + kept * b + 4 * c["c_out"], "flops": 2 * kept * c["m"]}
    ho, wo = _out(c)
    pixels = c["n"] * ho * wo
    if c["kind"] == "dw":
        b = 4 if c["dtype"] == "f32" else 2
        surv = c["c"] - int(round(c["prune"] * c["c"]))
        return {"bytes": (c["n"] * c["h"] * c["w"] + pixels) * c["c"] * b + surv * (4 * b + 2) + 4 * c["c"],
                "flops": 8 * surv * pixels}
    bx, bw, by = {"f32": (4, 4, 4), "f16": (2, 2, 2), "i8": (1, 1, 4)}[c["dtype"]]
    surv = _survivors(c)
    stored = pixels // (4 if c["pool"] else 1) * c["c_out"] * (1 if c["requant"] else by)
    nbytes = c["n"] * c["h"] * c["w"] * c["c_in"] * bx + surv * (4 * bw + 2) + 4 * c["c_out"] + stored
    nbytes += pixels * c["c_out"] * by if c["residual"] else 0
    nbytes += 4 * c["c_out"] if c["requant"] else 0
    return {"bytes": nbytes, "flops": 8 * surv * pixels}


def tolerance(case):
    """Integer layers are exact.  fp32: sums of up to a few thousand products in another order.
    fp16 storage: the fp32 sum is rounded once, so another order moves a result by one unit in
    the last place at most."""
    if case["dtype"] == "i8":
        return "exact"
    if case["dtype"] == "f32":
        return {"rel": 1e-5, "max": 1e-4}
    return {"rel": 1e-3, "max": 2e-3}


# --- inputs ------------------------------------------------------------------
def _activations(shape, dtype, g):
    """What a layer meets behind a ReLU: fp32 uniform on [0, 1), fp16 the positive half of a normal
    (half of it zeros), int8 uniform uint8 codes."""
    if dtype == "i8":
        return torch.randint(0, 256, shape, dtype=torch.uint8, device="cuda", generator=g)
    if dtype == "f32":
        return torch.rand(shape, device="cuda", generator=g)
    return torch.randn(shape, device="cuda", dtype=torch.float16, generator=g).clamp_(min=0)


def _weights(shape, dtype, sigma, g):
    if dtype == "i8":
        return torch.randint(-127, 128, shape, dtype=torch.int8, device="cuda", generator=g).cpu().numpy()
    return (torch.randn(shape, device="cuda", generator=g) * sigma).to(_T[dtype]).cpu().numpy()


def _patterns(count, prune, lib, g):
    """A pattern for every kernel, -1 for exactly the fraction `prune` of them, chosen at random."""
    pid = torch.randint(0, lib, (count,), dtype=torch.int16, device="cuda", generator=g)
    gone = torch.rand(count, device="cuda", generator=g).argsort()[:int(round(prune * count))]
    pid[gone] = -1
    return pid.cpu().numpy()


def _keep_flags(extent, block, others, rate, other_major, g):
    """Per pruning block `round(rate * size)` of its rows (or columns) kept, chosen at random."""
    blocks = -(-extent // block)
    flags = torch.zeros((blocks, others, block), dtype=torch.uint8, device="cuda")
    keys = torch.rand((blocks, others, block), device="cuda", generator=g)
    for part, size in ((slice(0, blocks - 1), block), (slice(blocks - 1, blocks), extent - (blocks - 1) * block)):
        flags[part].scatter_(-1, keys[part, :, :size].argsort(dim=-1)[..., :int(round(rate * size))], 1)
    flags = flags.transpose(0, 1) if other_major else flags
    return np.ascontiguousarray(flags.cpu().numpy())


def prepare(case, seed):
    c = case
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    dtype = c["dtype"]
    if c["kind"] == "gemm":
        m, k, co = c["m"], c["k"], c["c_out"]
        nbr, nbc = -(-co // c["br"]), -(-k // c["bc"])
        w = _weights((co, k), dtype, math.sqrt(2.0 / max(1.0, k * c["col_keep"])), g)
        layer = binding.BlockGemm(k, co, c["br"], c["bc"], dtype, w,
                                  _keep_flags(co, c["br"], nbc, c["row_keep"], False, g),
                                  _keep_flags(k, c["bc"], nbr, c["col_keep"], True, g))
        return {"case": c, "layer": layer, "x": _activations((m, k), dtype, g),
                "bias": torch.randn(co, device="cuda", generator=g) * 0.01,
                "y": torch.empty((m, co), dtype=_T[dtype], device="cuda")}
    masks = wl.pattern_library(c["lib"])
    ho, wo = _out(c)
    if c["kind"] == "dw":
        w = _weights((c["c"], 3, 3), dtype, math.sqrt(2.0 / 9.0), g)
        layer = binding.Depthwise(c["c"], c["stride"], dtype, masks, w, _patterns(c["c"], c["prune"], c["lib"], g))
        return {"case": c, "layer": layer, "x": _activations((c["n"], c["h"], c["w"], c["c"]), dtype, g),
                "bias": torch.randn(c["c"], device="cuda", generator=g) * 0.01,
                "y": torch.empty((c["n"], ho, wo, c["c"]), dtype=_T[dtype], device="cuda")}
    ci, co = c["c_in"], c["c_out"]
    w = _weights((co, ci, 3, 3), dtype, math.sqrt(2.0 / (9.0 * ci)), g)
    layer = binding.Packed(ci, co, c["stride"], dtype, masks, w, _patterns(co * ci, c["prune"], c["lib"], g))
    fused = bool(c["residual"] or c["pool"] or c["requant"])
    layer.plan(c["n"], c["h"], c["w"], no_small_blocks=fused)      # as the fused call wants it
    s = {"case": c, "layer": layer, "fused": fused, "residual": None, "scale": None,
         "x": _activations((c["n"], c["h"], c["w"], ci), dtype, g)}
    if dtype == "i8":
        s["bias"] = torch.randint(-(1 << 20), 1 << 20, (co,), dtype=torch.int32, device="cuda", generator=g)
    else:
        s["bias"] = torch.randn(co, device="cuda", generator=g) * 0.01
    out_t = torch.int32 if dtype == "i8" else _T[dtype]
    if c["residual"]:
        r = torch.randn((c["n"], ho, wo, co), device="cuda", generator=g)
        s["residual"] = (r * 2e5).to(torch.int32) if dtype == "i8" else (r * 0.5).to(out_t)
    if c["requant"]:                                               # codes spread over most of 0..255
        spread = math.sqrt(4.0 * _survivors(c) / co + 1.0) * 73.0 * 147.0 + 2 ** 19
        s["scale"] = (torch.rand(co, device="cuda", generator=g) + 0.5) * (80.0 / spread)
        out_t = torch.uint8
    if c["pool"]:
        ho, wo = ho // 2, wo // 2
    s["y"] = torch.empty((c["n"], ho, wo, co), dtype=out_t, device="cuda")
    return s


def run(state):
    s = state
    c, layer, y = s["case"], s["layer"], s["y"]
    stream = torch.cuda.current_stream().cuda_stream
    if c["kind"] == "gemm":
        layer.run(s["x"].data_ptr(), c["m"], s["bias"].data_ptr(), c["relu"], y.data_ptr(), stream)
    elif c["kind"] == "dw" or not s["fused"]:
        layer.run(s["x"].data_ptr(), c["n"], c["h"], c["w"], s["bias"].data_ptr(), c["relu"], y.data_ptr(), stream)
    else:
        layer.run_fused(s["x"].data_ptr(), c["n"], c["h"], c["w"], s["bias"].data_ptr(), y.data_ptr(), stream,
                        relu=c["relu"], pool=c["pool"],
                        residual_ptr=s["residual"].data_ptr() if c["residual"] else 0,
                        requant_scale_ptr=s["scale"].data_ptr() if c["requant"] else 0, zero_point=0)
    return y
