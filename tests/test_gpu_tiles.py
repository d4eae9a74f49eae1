"""Tiles and rounds of the convolution kernels at the sizes where their rules change: a last round in parts of the channels
(fp32 on the tensor cores), tiles of parts of strips (channel-innermost kernel)."""
import numpy as np
import pytest
import torch

import oracle
from paper_2608_20725_b200 import binding, workloads
from paper_2608_20725_b200.workloads import Layer
from gpu_helpers import check_conv, gpu_conv, gpu_conv_nhwc, oracle_inputs

pytestmark = pytest.mark.gpu


def L(name, N, C, H, W, Co, Kh, Kw, s, p, seed, xd="normal01"):
    return Layer(name, N, C, H, W, Co, Kh, Kw, s, p, seed, xd, "he_normal")


# 8.5 tiles of 128 positions an image; the tiles of the last round and the parts they go out in
@pytest.mark.parametrize("layer,bn", [
    (L("quarters", 18, 24, 32, 32, 256, 3, 3, 1, 1, 400), 256),       # 153 tiles: 5 in quarters
    (L("halves", 24, 24, 32, 32, 250, 3, 3, 1, 1, 401), 256),         # 204: 56 in halves, the last part not full
    (L("no_quarters", 18, 24, 32, 32, 150, 3, 3, 1, 1, 402), 160),    # 160 channels have halves, but no quarters of 16
    (L("whole", 26, 24, 32, 32, 120, 3, 3, 1, 1, 403), 128),          # 221: 73 in halves
    (L("whole2", 27, 24, 32, 32, 120, 3, 3, 1, 1, 404), 128)], ids=lambda v: getattr(v, "name", str(v)))     # 230: 82 whole
def test_f32_last_round_in_parts_of_the_channels(layer, bn, monkeypatch):
    monkeypatch.setenv("IM2WIN_F32_KERNEL", "split")
    monkeypatch.setenv("IM2WIN_F32_SPLIT_BN", str(bn))
    dims = layer.dims()
    assert binding.im2win_conv_kernel_name(dims, binding.F32) == "f32-split"
    x, f = workloads.make_small_integer_inputs(layer)
    y, _, _ = gpu_conv(x, f, dims, "f32")
    yr, _ = oracle.conv_direct(x.numpy(), f.numpy(), dims)
    assert np.array_equal(y.astype(np.float64), yr)
    # the sums of an output are those of any other round: the last image alone, in one round, gives the same bits
    x, f = workloads.make_inputs(layer)
    y, _, _ = gpu_conv(x, f, dims, "f32")
    monkeypatch.setenv("IM2WIN_F32_SPLIT_CTAS", "1")
    one, _, _ = gpu_conv(x[-1:], f, dict(dims, N=1), "f32")
    assert np.array_equal(y[-1:], one)
    yr, ar = oracle.conv_direct(x[-1:].numpy(), f.numpy(), dict(dims, N=1))
    check_conv(one, yr, ar, "f32", layer.name)


# reductions of 128 k-blocks of 64 and more, up to 256: strips of 28 in halves, 9 strips a tile; 27 and 30 do not divide
@pytest.mark.parametrize("layer", [
    L("k128", 1, 168, 28, 28, 72, 7, 7, 1, 3, 410), L("odd", 2, 165, 19, 27, 40, 7, 7, 1, 3, 411),
    L("thirds", 1, 120, 21, 30, 130, 9, 9, 1, 4, 412), L("wide", 1, 168, 9, 60, 64, 7, 7, 1, 3, 413),
    L("k256", 1, 256, 14, 28, 24, 8, 8, 1, 3, 414),
    L("short", 1, 160, 28, 28, 72, 7, 7, 1, 3, 415), L("strided", 1, 168, 28, 56, 72, 7, 7, 2, 3, 416)], ids=lambda l: l.name)
@pytest.mark.parametrize("layout", ["nchw", "nhwc"])
def test_nhwc_tiles_of_parts_of_strips(layer, layout, monkeypatch):
    monkeypatch.setenv("IM2WIN_NHWC_KERNEL", "overlap")
    dims = layer.dims()
    x, f = workloads.make_small_integer_inputs(layer)
    yr, _ = oracle.conv_direct(x.numpy(), f.numpy(), dims)
    y = gpu_conv_nhwc(x, f, dims, x_layout=layout)
    assert np.array_equal(np.asarray(y).astype(np.float64), yr)
    x, f = workloads.make_inputs(layer)
    y = gpu_conv_nhwc(x, f, dims, x_layout=layout)
    yr, ar = oracle.conv_direct(*oracle_inputs(x, f, "f16"), dims)
    check_conv(y, yr, ar, "f16", layer.name)
