"""The layers the library's speed is measured on, each run the way a program that uses it runs them.

A case is one convolution layer and the public calls that compute it (``paper_2608_20725_b200.binding``):

``form``
    ``layer``   im2win_transform, then the convolution of ``dtype``, on buffers the caller keeps
    ``call``    conv2d_im2win: the same from two tensors to a new output tensor
    ``nhwc``    im2win_transform_nhwc, then the channel-innermost convolution with its fused epilogue
    ``host``    im2win_layer_forward_host: page-locked host tensors in, a page-locked host tensor out
``static``
    the weights do not change between passes: the filter was packed once, beforehand (inference);
    otherwise the pass packs it (weights that are new each time)
``x_nhwc``, ``bias``, ``relu``, ``out16``, ``out_nhwc``
    (``nhwc`` only) the input's layout and the options of the epilogue
``dist``
    ``uniform01`` (what a ReLU leaves) or ``normal01`` (what a normalisation leaves)

Sizes are those of the library's benchmark layers (``workloads``) and, for odd and ragged ones, of no
network in particular.  Every pass writes the whole window tensor and the whole output; both are returned.
"""
import math

import torch

from paper_2608_20725_b200 import binding


def _case(name, form, dtype, N, C, H, W, Co, K, stride, pad, dist, **options):
    c = {"name": name, "form": form, "dtype": dtype, "N": N, "C": C, "H": H, "W": W, "Co": Co, "Kh": K, "Kw": K,
         "stride": stride, "pad": pad, "dist": dist, "static": False, "x_nhwc": False, "bias": False, "relu": False,
         "out16": False, "out_nhwc": False}
    unknown = set(options) - set(c)
    assert not unknown, unknown
    c.update(options)
    return c


def listed():
    return [
        # the smallest call: one small image, tensors in, tensor out; launches and host time are all of it
        _case("tiny_f32_call", "call", "f32", 1, 3, 32, 32, 16, 3, 1, 1, "normal01"),
        # one image through a middle layer of a network kept channel-innermost: latency of serving a single request
        _case("one_image_f16_nhwc", "nhwc", "f16", 1, 64, 56, 56, 64, 3, 1, 1, "uniform01", static=True, x_nhwc=True,
              bias=True, relu=True, out16=True, out_nhwc=True),
        # the ordinary 3x3 layer of a residual network at batch 128, once in each precision, weights packed in the pass
        _case("ordinary_3x3_f32", "layer", "f32", 128, 64, 56, 56, 64, 3, 1, 1, "uniform01"),
        _case("ordinary_3x3_f16", "layer", "f16", 128, 64, 56, 56, 64, 3, 1, 1, "uniform01"),
        # the network's first layer: three channels, a large kernel, stride 2, output-bound
        _case("stem_7x7_f16", "layer", "f16", 128, 3, 224, 224, 64, 7, 2, 3, "normal01", static=True),
        # down-sampling layer between two stages (stride 2, odd plane pitch)
        _case("down_3x3_f16", "layer", "f16", 128, 256, 28, 28, 512, 3, 2, 1, "uniform01", static=True),
        # deep layer on tiny images, fp32 inference with packed weights: few positions, long reduction
        _case("deep_7x7_image_f32", "layer", "f32", 128, 512, 7, 7, 512, 3, 1, 1, "uniform01", static=True),
        # deep layer of a channel-innermost network, from NCHW data, fp32 output
        _case("deep_14x14_image_f16_nhwc", "nhwc", "f16", 128, 256, 14, 14, 256, 3, 1, 1, "uniform01", static=True),
        # wide kernel in a channel-innermost chain, fused epilogue, the largest fp16 product
        _case("wide_7x7_f16_nhwc", "nhwc", "f16", 64, 256, 28, 28, 256, 7, 1, 3, "normal01", static=True, x_nhwc=True,
              bias=True, relu=True, out16=True, out_nhwc=True),
        # the largest fp32 reduction of the kernel-size sweep
        _case("wide_11x11_f32", "layer", "f32", 64, 256, 28, 28, 256, 11, 1, 5, "normal01"),
        # nothing is a round number: odd image, channel counts that fill no tile, stride 2
        _case("ragged_5x5_f32", "layer", "f32", 13, 37, 45, 61, 75, 5, 2, 2, "normal01"),
        # a layer applied to data that lives in host memory
        _case("from_host_f16", "host", "f16", 32, 64, 56, 56, 64, 3, 1, 1, "uniform01"),
    ]


# The largest listed case bounds the drawn ones, in seconds at these rates (fp32 and fp16 FLOP/s, bytes/s).
_RATE = {"f32": 5e13, "f16": 5e14}
_BYTES = 4e12
_HOST_BYTES = 2e10
_MOST_SECONDS = 6e-3


def _out(c):
    return ((c["H"] + 2 * c["pad"] - c["Kh"]) // c["stride"] + 1, (c["W"] + 2 * c["pad"] - c["Kw"]) // c["stride"] + 1)


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    while True:
        form, dtype = rng.choice([("layer", "f32")] * 4 + [("layer", "f16")] * 4 + [("nhwc", "f16")] * 4
                                 + [("call", "f32"), ("call", "f16"), ("host", "f32"), ("host", "f16")])
        kh = kw = rng.choice([1, 3, 3, 3, 3, 5, 7, 11])
        if rng.random() < 0.1:
            kw = rng.choice([1, 3, 5, 7])                           # kernels that are not square
        stride = rng.choice([1, 1, 1, 1, 2, 2, 4 if kh >= 7 else 1])
        pad = rng.choice([0, (kh - 1) // 2, (kh - 1) // 2])
        h = _log_int(rng, 7, 224)
        w = h if rng.random() < 0.7 else _log_int(rng, 7, 224)
        channels = [rng.choice([3, 3, 8, 16, 32, 64, 64, 96, 128, 128, 256, 256, 512]), _log_int(rng, 3, 512)]
        c_in = rng.choice(channels)
        c_out = rng.choice([rng.choice([16, 32, 64, 64, 96, 128, 128, 256, 256, 512]), _log_int(rng, 8, 512)])
        n = rng.choice([1, 2, 4, 8, 16, 32, 64, 128, _log_int(rng, 1, 160)])
        if min(h, w) + 2 * pad < max(kh, kw):
            continue
        c = _case("", form, dtype, n, c_in, h, w, c_out, kh, stride, pad, rng.choice(["uniform01", "normal01"]))
        c["Kw"] = kw
        if form in ("layer", "nhwc"):
            c["static"] = rng.random() < 0.5
        if form == "nhwc":
            for option in ("x_nhwc", "bias", "relu", "out16", "out_nhwc"):
                c[option] = rng.random() < 0.5
        if min(_out(c)) < 1:
            continue
        need = work(c)
        seconds = need["flops"] / _RATE[dtype] + need["bytes"] / (_HOST_BYTES if form == "host" else _BYTES)
        if seconds > _MOST_SECONDS or need["bytes"] > 1.2e9:
            continue
        del c["name"]
        return c


def _dims(c):
    return {k: c[k] for k in ("N", "C", "H", "W", "Co", "Kh", "Kw", "stride", "pad")}


def prepare(case, seed):
    dims = _dims(case)
    tdt = torch.float32 if case["dtype"] == "f32" else torch.float16
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    xs = (case["N"], case["C"], case["H"], case["W"])
    x = (torch.rand if case["dist"] == "uniform01" else torch.randn)(xs, generator=g, device="cuda")
    std = math.sqrt(2.0 / (case["C"] * case["Kh"] * case["Kw"]))
    f = torch.randn((case["Co"], case["C"], case["Kh"], case["Kw"]), generator=g, device="cuda") * std
    x, f = x.to(tdt), f.to(tdt)
    s = {"case": case, "shape": binding.as_shape(dims), "x": x, "f": f}
    if case["form"] == "layer":
        s["window"], s["scratch"], s["y"] = binding.alloc_layer_buffers(dims, tdt)
        if case["static"]:
            binding.im2win_pack_filter(f, s["scratch"], s["shape"])
    elif case["form"] == "nhwc":
        if case["x_nhwc"]:
            s["x"] = x.permute(0, 2, 3, 1).contiguous()
        out = torch.float16 if case["out16"] else torch.float32
        layout = binding.NHWC if case["out_nhwc"] else binding.NCHW
        s["bias"] = torch.randn(case["Co"], generator=g, device="cuda") * 0.5 if case["bias"] else None
        s["epilogue"] = binding.make_epilogue(s["bias"], case["relu"], out, layout)
        s["window"], s["scratch"], s["y"] = binding.alloc_nhwc_buffers(dims, out, layout)
        if case["static"]:
            binding.im2win_pack_filter_nhwc(f, s["scratch"], s["shape"])
    elif case["form"] == "host":
        code = binding.F32 if case["dtype"] == "f32" else binding.F16
        s["x"] = torch.empty(x.shape, dtype=tdt, pin_memory=True).copy_(x)
        s["f"] = torch.empty(f.shape, dtype=tdt, pin_memory=True).copy_(f)
        s["y"] = torch.empty((case["N"], case["Co"]) + _out(case), dtype=torch.float32, pin_memory=True)
        s["workspace"] = torch.empty(binding.im2win_layer_workspace_size(dims, code), dtype=torch.uint8, device="cuda")
    return s


def run(state):
    case, shape = state["case"], state["shape"]
    form = case["form"]
    if form == "call":
        return binding.conv2d_im2win(state["x"], state["f"], case["stride"], case["pad"])
    if form == "host":
        binding.im2win_layer_forward_host(state["x"], state["f"], state["y"], state["workspace"], shape)
        return state["y"]
    window, scratch, y = state["window"], state["scratch"], state["y"]
    if form == "layer":
        binding.im2win_transform(state["x"], window, shape)
        if case["static"]:
            binding.im2win_conv_packed(window, y, scratch, shape)
        elif case["dtype"] == "f32":
            binding.im2win_conv_f32(window, state["f"], y, scratch, shape)
        else:
            binding.im2win_conv_f16(window, state["f"], y, scratch, shape)
    else:
        binding.im2win_transform_nhwc(state["x"], binding.NHWC if case["x_nhwc"] else binding.NCHW, window, shape)
        if case["static"]:
            binding.im2win_conv_packed_nhwc(window, y, scratch, shape, state["epilogue"])
        else:
            binding.im2win_conv_f16_nhwc(window, state["f"], y, scratch, shape, state["epilogue"])
    return {"window": window, "y": y}


def work(case):
    """Input, filter and output once; the window tensor written by the one call and read by the other, where
    the caller holds it (``call`` and ``host`` keep it to themselves)."""
    ho, wo = _out(case)
    es = 4 if case["dtype"] == "f32" else 2
    c, rows = case["C"], case["N"] * ho
    x = case["N"] * c * case["H"] * case["W"] * es
    f = case["Co"] * c * case["Kh"] * case["Kw"] * es
    y = rows * wo * case["Co"] * (2 if case["out16"] else 4)
    stored = (c + 7) // 8 * 8 if case["form"] == "nhwc" else c
    window = rows * stored * case["Kh"] * (case["W"] + 2 * case["pad"]) * es
    moved = x + f + y + (2 * window if case["form"] in ("layer", "nhwc") else 0)
    return {"bytes": moved, "flops": 2 * rows * wo * case["Co"] * c * case["Kh"] * case["Kw"]}


def tolerance(case):
    """About four times the distance from the same layer in 64 bits, over the listed and many drawn cases: fp32
    3e-6 (largest element 2e-5), fp16 products in fp32 sums 7e-6 (2.2e-5), binary16 stores 2.1e-4 (5.1e-4)."""
    if case["out16"]:
        return {"rel": 8e-4, "max": 2e-3}
    if case["dtype"] == "f16":
        return {"rel": 3e-5, "max": 1e-4}
    return {"rel": 1e-5, "max": 8e-5}
