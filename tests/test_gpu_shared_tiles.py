"""Tiles whose reduction the CTAs of a cluster share: every form of the shifted-view and the run-staged fp16 kernel and of the fp32
tensor-core kernel, parts that start inside an octet of channels or a raw slot, numbers of CTAs that divide neither the k-blocks nor
the channels, shares without a channel; and which layers are shared.

Tolerances: those of gpu_helpers (the sum of a part is an fp32 accumulator's, and up to 16 of them are added in fp32); integer-valued
inputs exactly.
"""
import ctypes

import numpy as np
import pytest
import torch

import oracle
from paper_2608_20725_b200 import binding, workloads
from paper_2608_20725_b200.workloads import Layer
from gpu_helpers import check_conv, gpu_conv, oracle_inputs, runs_form, split_form


def L(name, N, C, H, W, Co, Kh, Kw, s, p, seed, xd="normal01"):
    return Layer(name, N, C, H, W, Co, Kh, Kw, s, p, seed, xd, "he_normal")


def tile_ctas(dims):
    """CTAs that share the reduction of a tile in the kernel that an fp16 layer takes.  Needs no GPU."""
    fn = binding.lib().im2win_f16_tile_ctas
    fn.argtypes, fn.restype = [ctypes.POINTER(binding.Shape)], ctypes.c_int32
    return fn(ctypes.byref(binding.as_shape(dims)))


def compare(layer, precision):
    dims = layer.dims()
    x, f = workloads.make_small_integer_inputs(layer)
    y, _, _ = gpu_conv(x, f, dims, precision)
    yr, _ = oracle.conv_direct(x.numpy(), f.numpy(), dims)
    assert np.array_equal(y.astype(np.float64), yr)
    x, f = workloads.make_inputs(layer)
    y, _, _ = gpu_conv(x, f, dims, precision)
    yr, ar = oracle.conv_direct(*oracle_inputs(x, f, precision), dims)
    check_conv(y, yr, ar, precision, layer.name)
    again, _, _ = gpu_conv(x, f, dims, precision)            # the parts are added in one order
    assert np.array_equal(y, again)


# (channel tile, CTAs); 64, 128 and 256 channels, one to three column classes' worth of staged chunks
@pytest.mark.gpu
@pytest.mark.parametrize("layer,bn,ctas", [
    (L("c300", 2, 75, 9, 9, 300, 3, 3, 1, 1, 600), 256, 4), (L("c300_64", 2, 75, 9, 9, 300, 3, 3, 1, 1, 600), 64, 3),
    (L("c130", 3, 90, 7, 10, 130, 5, 5, 1, 2, 601), 128, 8), (L("c9", 4, 130, 6, 6, 9, 3, 3, 1, 1, 602), 64, 7),
    (L("c9_16", 1, 350, 6, 6, 9, 3, 3, 1, 1, 603), 64, 16),          # more CTAs than channels: shares without one
    (L("s2", 2, 100, 17, 13, 70, 3, 3, 2, 1, 604), 128, 5), (L("s2_256", 1, 64, 15, 15, 200, 7, 7, 2, 3, 605), 256, 6),
    (L("s3", 1, 60, 20, 23, 40, 4, 5, 3, 0, 606), 64, 2), (L("k1x7", 3, 129, 5, 12, 66, 1, 7, 1, 0, 607), 128, 3)],
    ids=lambda v: getattr(v, "name", str(v)))
def test_shifted_view_tiles(layer, bn, ctas, monkeypatch):
    monkeypatch.setenv("IM2WIN_F16_KERNEL", "shift")
    monkeypatch.setenv("IM2WIN_F16_SHIFT_BN", str(bn))
    monkeypatch.setenv("IM2WIN_F16_SPLIT", str(ctas))
    assert binding.im2win_conv_kernel_name(layer.dims(), binding.F16) == "f16-shift" and tile_ctas(layer.dims()) == ctas
    compare(layer, "f16")


# (staging mode, CTAs): elements, words of two, pairs of rows, unit by unit
@pytest.mark.gpu
@pytest.mark.parametrize("layer,mode,ctas", [
    (L("rows", 2, 130, 14, 12, 130, 3, 3, 1, 1, 610), 2, 3), (L("rows_7", 1, 200, 14, 12, 40, 3, 3, 1, 1, 611), 2, 7),
    (L("words", 2, 72, 28, 28, 100, 3, 3, 2, 1, 612), 1, 5), (L("words_12", 1, 150, 20, 20, 9, 5, 5, 2, 2, 613), 1, 12),
    (L("elements", 3, 90, 13, 15, 48, 3, 3, 1, 1, 614), 0, 4), (L("elements_9", 2, 64, 30, 31, 180, 3, 3, 3, 0, 615), 0, 9),
    (L("units", 2, 40, 16, 12, 48, 5, 5, 1, 2, 616), 3, 3), (L("units_1x1", 2, 520, 8, 16, 33, 1, 1, 1, 0, 617), 3, 4),
    (L("units_2el", 2, 100, 20, 28, 40, 1, 2, 2, 0, 618), 3, 3),    # two octets a slot: parts start within one
    (L("units_quad", 1, 3, 60, 60, 20, 11, 11, 4, 2, 619), 3, 3),   # up to four channels: one slot for all parts
    (L("units_11", 1, 48, 20, 20, 24, 11, 11, 2, 5, 620), 3, 16)], ids=lambda v: getattr(v, "name", str(v)))
def test_run_staged_tiles(layer, mode, ctas, monkeypatch):
    monkeypatch.setenv("IM2WIN_F16_KERNEL", "runs")
    monkeypatch.setenv("IM2WIN_F16_SPLIT", str(ctas))
    dims = layer.dims()
    assert binding.im2win_conv_kernel_name(dims, binding.F16) == "f16-runs" and tile_ctas(dims) == ctas
    assert runs_form(dims).mode == mode and not runs_form(dims).pair
    compare(layer, "f16")
    # an infinity and a NaN reach exactly the outputs whose windows hold them
    x, f = workloads.make_inputs(layer)
    x = x.clone()
    x.view(-1)[x.numel() // 3] = float("inf")
    x.view(-1)[x.numel() // 2] = float("nan")
    y, _, _ = gpu_conv(x, f, dims, "f16")
    ref = torch.nn.functional.conv2d(x.half().double(), f.half().double(), stride=layer.stride, padding=layer.pad).numpy()
    assert np.array_equal(np.isfinite(y), np.isfinite(ref)) and np.array_equal(np.isnan(y), np.isnan(ref))


@pytest.mark.gpu
@pytest.mark.parametrize("layer,form", [
    (L("f64", 2, 120, 9, 9, 64, 3, 3, 1, 1, 630), (64, 5)), (L("f64_16", 1, 350, 6, 6, 40, 3, 3, 1, 1, 631), (48, 16)),
    (L("f128", 1, 150, 8, 11, 100, 3, 3, 2, 1, 632), (112, 9)), (L("f256", 1, 100, 9, 9, 250, 3, 5, 1, 1, 633), (256, 3)),
    (L("f16", 1, 100, 9, 9, 7, 3, 3, 2, 1, 634), (16, 10))], ids=lambda v: getattr(v, "name", str(v)))
def test_fp32_tiles(layer, form, monkeypatch):
    monkeypatch.setenv("IM2WIN_F32_KERNEL", "split")
    monkeypatch.setenv("IM2WIN_F32_SPLIT_BN", str(form[0]))
    monkeypatch.setenv("IM2WIN_F32_SPLIT_CTAS", str(form[1]))
    assert split_form(layer.dims())[:2] == form
    compare(layer, "f32")
    # outputs that are not finite are computed again, by the CTA that finishes their channel
    x, f = workloads.make_inputs(layer)
    x = x.clone()
    x.view(-1)[x.numel() // 3] = float("inf")
    x.view(-1)[x.numel() // 2] = float("nan")
    y, _, _ = gpu_conv(x, f, layer.dims(), "f32")
    monkeypatch.setenv("IM2WIN_F32_KERNEL", "ffma")
    z, _, _ = gpu_conv(x, f, layer.dims(), "f32")
    odd = ~np.isfinite(z)
    assert odd.any() and np.array_equal(np.isnan(y), np.isnan(z)) and np.array_equal(y[odd & ~np.isnan(z)], z[odd & ~np.isnan(z)])
    assert np.isfinite(y[~odd]).all()


# a wait of one CTA runs out: the others of its cluster return as well, and the next call is exact
@pytest.mark.gpu
def test_a_cta_that_gives_up_holds_up_no_other(monkeypatch):
    monkeypatch.setenv("IM2WIN_F16_KERNEL", "runs")
    monkeypatch.setenv("IM2WIN_F16_SPLIT", "3")
    layer = L("wait_shared", 2, 130, 14, 12, 130, 3, 3, 1, 1, 640)
    dims = layer.dims()
    x, f = workloads.make_inputs(layer)
    want, _, _ = gpu_conv(x, f, dims, "f16")
    xd, fd = x.half().cuda(), f.half().cuda()
    window, scratch, y = binding.alloc_layer_buffers(dims, torch.float16)
    binding.im2win_transform(xd, window, dims)
    binding.im2win_pack_filter(fd, scratch, dims)
    torch.cuda.synchronize()
    words = scratch[:256].view(torch.int32)
    words[1] = 4096
    words[2] = 0x0d0a11fe
    binding.im2win_conv_packed(window, y, scratch, dims)
    with pytest.raises(binding.Im2winError) as err:
        binding.im2win_check_status(scratch)
    assert err.value.code == 7
    binding.im2win_conv_f16(window, fd, y, scratch, dims)
    binding.im2win_check_status(scratch)
    assert np.array_equal(y.cpu().numpy(), want)


# parts of a batch are added up as the whole batch is, whatever clusters they would take alone
@pytest.mark.gpu
@pytest.mark.parametrize("layer", [L("host_shift", 32, 256, 19, 19, 16, 7, 7, 1, 3, 650), L("host_runs", 24, 512, 15, 15, 128, 3, 3, 2, 1, 651),
                                   L("host_alone", 64, 256, 19, 19, 65, 3, 3, 1, 1, 652)], ids=lambda l: l.name)
def test_host_call_in_parts(layer):
    dims = layer.dims()
    x, f = workloads.make_inputs(layer)
    y, _, _ = gpu_conv(x, f, dims, "f16")
    out = torch.full(y.shape, float("nan")).pin_memory()
    ws = torch.empty(binding.im2win_layer_workspace_size(dims, binding.F16), dtype=torch.uint8, device="cuda")
    binding.im2win_layer_forward_host(x.half().pin_memory(), f.half().pin_memory(), out, ws, dims)
    torch.cuda.synchronize()
    assert np.array_equal(out.numpy(), y)


@pytest.mark.parametrize("layer,ctas", [
    ((27, 512, 15, 15, 128, 3, 3, 2, 1), 6),         # run-staged, 16 tiles of 24 k-blocks
    ((4, 256, 18, 18, 256, 7, 7, 2, 3), 10),         # shifted views
    ((16, 256, 115, 10, 80, 3, 5, 2, 1), 2),         # 44 tiles: 45 clusters of three fit an idle GPU, 42 one that is being left
    ((8, 86, 36, 36, 128, 11, 11, 2, 5), 4),         # 26 tiles, likewise 26 and 25 clusters of five
    ((1, 64, 50, 50, 104, 3, 3, 1, 0), 1),           # too little to share
    ((128, 64, 56, 56, 64, 3, 3, 1, 1), 1),          # tiles enough
    ((8, 393, 9, 20, 128, 11, 11, 2, 5), 1)])        # 47553 terms
def test_which_fp16_layers_are_shared(layer, ctas):
    assert tile_ctas(layer) == ctas


@pytest.mark.parametrize("layer,form", [
    ((2, 256, 35, 35, 78, 7, 7, 1, 0), (48, 4)),     # 16 tiles: only 15 clusters of 8 are resident at once
    ((2, 256, 36, 36, 23, 11, 11, 1, 5), (32, 4)),   # 26 tiles: no fives
    ((4, 512, 14, 14, 90, 11, 11, 4, 5), (16, 16)),
    ((1, 256, 8, 8, 103, 3, 3, 1, 0), (16, 12))])
def test_which_fp32_layers_are_shared(layer, form):
    assert split_form(layer)[:2] == form


# kernels that start before the one ahead of them has ended (transform, filter pack, convolution): passes queued back to back on the same
# window and scratch, inputs and filters in turn, give what each gives alone
@pytest.mark.gpu
@pytest.mark.parametrize("layer,dtype,kernel", [
    (L("b_split", 8, 64, 30, 30, 64, 3, 3, 1, 1, 660), torch.float32, "f32-split"), (L("b_ffma", 8, 3, 40, 40, 40, 3, 3, 1, 1, 661), torch.float32, "f32-ffma"),
    (L("b_runs", 16, 64, 28, 28, 64, 3, 3, 1, 1, 662), torch.float16, "f16-runs"), (L("b_shift", 2, 128, 21, 21, 64, 7, 7, 1, 3, 663), torch.float16, "f16-shift"),
    (L("b_stem", 16, 3, 60, 60, 64, 7, 7, 2, 3, 664), torch.float16, "f16-stem"), (L("b_mat", 8, 128, 28, 28, 256, 3, 3, 1, 1, 665), torch.float16, "f16-mat"),
    (L("b_nhwc", 8, 40, 30, 30, 70, 3, 3, 1, 1, 666), torch.float16, None)], ids=lambda v: getattr(v, "name", str(v)))
def test_passes_back_to_back(layer, dtype, kernel):
    dims = layer.dims()
    code = binding.F32 if dtype == torch.float32 else binding.F16
    assert kernel is None or binding.im2win_conv_kernel_name(dims, code) == kernel
    x, f = workloads.make_inputs(layer)
    xs, fs = [x.to(dtype).cuda(), (x.flip(0) * 2).to(dtype).cuda()], [f.to(dtype).cuda(), f.flip(0).to(dtype).cuda()]
    window, scratch, y = binding.alloc_layer_buffers(dims, dtype) if kernel else binding.alloc_nhwc_buffers(dims)
    out = [torch.empty_like(y) for _ in range(12)]

    def one(i, y):
        if kernel is None:
            binding.im2win_transform_nhwc(xs[i % 2], binding.NCHW, window, dims)
            binding.im2win_conv_f16_nhwc(window, fs[i % 3 % 2], y, scratch, dims)
        else:
            binding.im2win_transform(xs[i % 2], window, dims)
            (binding.im2win_conv_f32 if code == binding.F32 else binding.im2win_conv_f16)(window, fs[i % 3 % 2], y, scratch, dims)

    for i in range(12):
        one(i, out[i])
    binding.im2win_check_status(scratch)
    for i in range(12):
        one(i, y)
        binding.im2win_check_status(scratch)
        assert torch.equal(out[i], y)
