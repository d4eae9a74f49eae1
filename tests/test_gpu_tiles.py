"""Tiles and rounds of the convolution kernels at the sizes where their rules change: a last round in parts of the channels
(fp32 on the tensor cores), tiles of parts of strips (channel-innermost kernel), the ways the run-staged kernel brings
its columns in."""
from dataclasses import replace

import numpy as np
import pytest
import torch

import oracle
from paper_2608_20725_b200 import binding, workloads
from paper_2608_20725_b200.workloads import Layer
from gpu_helpers import check_conv, gpu_conv, gpu_conv_nhwc, oracle_inputs, runs_form

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


# reductions of 128 k-blocks of 64 and more, up to 256: strips of 28 in halves, 9 strips a tile; 27 and 50 do not divide
@pytest.mark.parametrize("layer", [
    L("k128", 5, 168, 28, 28, 72, 7, 7, 1, 3, 410), L("odd", 5, 165, 19, 27, 40, 7, 7, 1, 3, 411),
    L("w36", 4, 120, 21, 36, 130, 9, 9, 1, 4, 412), L("w50", 4, 168, 9, 50, 64, 7, 7, 1, 3, 413),
    L("k256", 5, 256, 14, 28, 24, 8, 8, 1, 3, 414),
    L("short", 5, 160, 28, 28, 24, 7, 7, 1, 3, 415), L("strided", 5, 168, 28, 56, 24, 7, 7, 2, 3, 416)], ids=lambda l: l.name)
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


# the columns of the run-staged kernel: elements, words of two, pairs of rows, unit by unit; copies of one, two, four and eight
# channels; CTA pairs.  (form: staging mode, pairs, planes of a tiled copy's row)
@pytest.mark.parametrize("layer,form", [
    (L("pairs_1", 2, 48, 20, 14, 150, 3, 3, 1, 1, 420), (2, 1, 1)),    # CTA pairs, an odd number of position tiles
    (L("pairs_4", 3, 28, 14, 11, 33, 3, 3, 1, 1, 421), (2, 0, 4)),     # half an octet in the last slot, two images in a tile
    (L("pairs_18", 2, 18, 13, 12, 70, 3, 3, 1, 1, 422), (2, 0, 0)),    # four planes, but no multiple of four channels: bulk copies
    (L("pairs_s", 5, 40, 9, 8, 16, 3, 3, 1, 0, 423), (2, 0, 0)),       # several images in a tile: bulk copies
    (L("words_2", 3, 40, 28, 28, 150, 3, 3, 2, 1, 424), (1, 1, 2)),    # stride 2, CTA pairs, an odd number of position tiles
    (L("words_c33", 2, 33, 28, 28, 300, 3, 3, 2, 1, 425), (1, 1, 0)),  # an odd number of channels; pairs, two channel tiles, the last not full
    (L("words_10", 1, 24, 30, 30, 40, 5, 5, 2, 1, 426), (1, 0, 0)),    # ten elements a column, boxes too wide
    (L("words_2el", 1, 24, 30, 28, 40, 1, 2, 2, 0, 427), (3, 0, 2)),   # two elements, two octets a slot
    (L("halves_5", 2, 16, 16, 12, 48, 5, 5, 1, 2, 428), (3, 0, 1)),    # five elements, four rows below the tile
    (L("halves_1", 2, 520, 16, 16, 220, 1, 1, 1, 0, 429), (3, 1, 1)),  # one element, four octets a slot, the last slot not full; pairs
    (L("halves_odd", 2, 40, 13, 15, 48, 3, 3, 1, 1, 430), (0, 0, 0)),  # an odd number of columns in an image; eight planes
    (L("halves_9", 3, 64, 30, 31, 180, 3, 3, 3, 0, 433), (0, 1, 0)),   # stride 3, CTA pairs, an odd number of position tiles
    (L("last_pair", 9, 48, 16, 14, 256, 3, 3, 1, 1, 431), (2, 1, 1)),  # 18 position tiles
    (L("rounds", 32, 48, 20, 30, 250, 3, 3, 1, 1, 432), (2, 1, 1))],   # more pairs than the GPU holds, the channel tile not full
    ids=lambda v: getattr(v, "name", None))
@pytest.mark.parametrize("tiled,pair,units", [("1", "1", None), ("0", "1", None), ("1", "0", None), ("1", "1", "1"), ("1", "1", "0")])
def test_f16_runs_columns_and_copies(layer, form, tiled, pair, units, monkeypatch):
    monkeypatch.setenv("IM2WIN_F16_KERNEL", "runs")
    monkeypatch.setenv("IM2WIN_F16_RUNS_TILED", tiled)
    monkeypatch.setenv("IM2WIN_F16_PAIR", pair)
    if units:
        monkeypatch.setenv("IM2WIN_F16_RUNS_UNITS", units)
    dims = layer.dims()
    assert binding.im2win_conv_kernel_name(dims, binding.F16) == "f16-runs"
    got = runs_form(dims)
    assert (got.mode == 3) == (form[0] == 3 if units is None else units == "1") and (units or got.mode == form[0])
    assert got.pair == form[1] * int(pair) and got.planes == form[2] * int(tiled)
    assert layer.name != "rounds" or got.ntm > 148
    x, f = workloads.make_small_integer_inputs(layer)
    y, _, _ = gpu_conv(x, f, dims, "f16")
    yr, _ = oracle.conv_direct(x.numpy(), f.numpy(), dims)
    assert np.array_equal(y.astype(np.float64), yr)
    x, f = workloads.make_inputs(layer)
    y, _, _ = gpu_conv(x, f, dims, "f16")
    yr, ar = oracle.conv_direct(*oracle_inputs(x, f, "f16"), dims)
    check_conv(y, yr, ar, "f16", layer.name)
    # an infinity and a NaN reach exactly the outputs whose windows hold them
    x.view(-1)[x.numel() // 3] = float("inf")
    x.view(-1)[x.numel() // 2] = float("nan")
    y, _, _ = gpu_conv(x, f, dims, "f16")
    ref = torch.nn.functional.conv2d(x.half().double(), f.half().double(), stride=layer.stride, padding=layer.pad).numpy()
    assert np.array_equal(np.isfinite(y), np.isfinite(ref)) and np.array_equal(np.isnan(y), np.isnan(ref))


# Four teams of staging warps on rings of four raw slots and of eight, which go round two to eight times in a tile
@pytest.mark.parametrize("layer,slots", [
    (L("teams_128", 3, 128, 28, 28, 128, 3, 3, 1, 1, 440), 4), (L("teams_64", 1, 64, 48, 50, 128, 3, 3, 1, 0, 441), 4),
    (L("teams_pair", 2, 256, 20, 20, 256, 3, 3, 1, 1, 442), 4), (L("teams_to_64", 2, 128, 56, 30, 64, 3, 3, 1, 1, 443), 4),
    (L("teams_eight", 2, 160, 30, 30, 16, 3, 3, 1, 1, 444), 8)], ids=lambda v: getattr(v, "name", str(v)))
def test_f16_runs_teams_on_their_slots(layer, slots, monkeypatch):
    monkeypatch.setenv("IM2WIN_F16_KERNEL", "runs")
    dims = layer.dims()
    form = runs_form(dims)
    assert (form.mode, form.teams, form.slots) == (2, 4, slots) and layer.C // 8 >= 2 * slots
    for seed in range(3):                                    # (new buffers every time: cold copies)
        x, f = workloads.make_small_integer_inputs(replace(layer, seed=layer.seed + 100 * seed))
        y, _, _ = gpu_conv(x, f, dims, "f16")
        yr, _ = oracle.conv_direct(x.numpy(), f.numpy(), dims)
        assert np.array_equal(y.astype(np.float64), yr)


# Rows below the tile: as many as a warp reads for a whole group of three or six units (ten, five), and more, which only the form
# that goes unit by unit takes
@pytest.mark.parametrize("layer,mode,halo", [
    (L("low_13", 1, 24, 16, 20, 24, 13, 13, 1, 6, 450), 3, 12), (L("low_pair", 2, 40, 14, 17, 150, 13, 14, 1, 3, 451), 3, 13),
    (L("low_quad", 1, 3, 18, 21, 16, 12, 12, 1, 2, 452), 3, 11), (L("low_31", 1, 72, 6, 40, 16, 1, 32, 1, 0, 457), 3, 31),
    (L("low_11", 1, 20, 15, 20, 20, 12, 12, 1, 3, 458), 3, 11), (L("low_3x12", 1, 40, 14, 20, 48, 3, 12, 1, 2, 456), 3, 11),
    (L("low_3x11", 1, 40, 14, 20, 48, 3, 11, 1, 2, 459), 2, 10), (L("low_10", 2, 24, 14, 16, 33, 10, 10, 1, 4, 453), 0, 9),
    (L("low_6", 1, 20, 20, 15, 150, 10, 7, 1, 3, 454), 0, 6), (L("low_5", 1, 20, 20, 15, 150, 10, 6, 1, 3, 460), 1, 5),
    (L("low_s2", 1, 24, 15, 32, 20, 5, 15, 2, 2, 455), 0, 7)], ids=lambda v: getattr(v, "name", str(v)))
def test_f16_runs_rows_below_the_tile(layer, mode, halo, monkeypatch):
    monkeypatch.setenv("IM2WIN_F16_KERNEL", "runs")
    monkeypatch.setenv("IM2WIN_F16_RUNS_UNITS", "0")
    dims = layer.dims()
    form = runs_form(dims)
    assert (form.mode, form.halo) == (mode, halo)
    x, f = workloads.make_small_integer_inputs(layer)
    y, _, _ = gpu_conv(x, f, dims, "f16")
    yr, _ = oracle.conv_direct(x.numpy(), f.numpy(), dims)
    assert np.array_equal(y.astype(np.float64), yr)
    x, f = workloads.make_inputs(layer)
    y, _, _ = gpu_conv(x, f, dims, "f16")
    yr, ar = oracle.conv_direct(*oracle_inputs(x, f, "f16"), dims)
    check_conv(y, yr, ar, "f16", layer.name)
