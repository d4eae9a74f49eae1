"""Channel-innermost rows stored through shared memory (channels that are no whole number of 16-byte vectors) and by ragged numbers of
vectors: rows that start on odd halves, last chunks of 1 to 31 channels, tiles whose strips leave gaps, tiles of parts of strips, several
channel tiles, a short last round whose tiles several CTAs share; tiles shared by clusters.  Integer-valued inputs exactly (the result is one
fp32 sum, rounded once), guard bands around the output.
"""
import functools

import numpy as np
import pytest

import oracle
from paper_2608_20725_b200 import binding, workloads
from paper_2608_20725_b200.workloads import Layer
from gpu_helpers import check_conv, gpu_conv_nhwc, oracle_inputs

pytestmark = pytest.mark.gpu


def L(name, N, C, H, W, Co, Kh, Kw, s, p, seed):
    return Layer(name, N, C, H, W, Co, Kh, Kw, s, p, seed, "normal01", "he_normal")


@pytest.mark.parametrize("kernel", ["shift", "overlap"])
@pytest.mark.parametrize("layer", [
    L("c1", 3, 8, 9, 11, 1, 3, 3, 1, 1, 700), L("c7", 2, 8, 12, 9, 7, 3, 3, 1, 0, 701), L("c9", 2, 16, 10, 10, 9, 1, 1, 1, 0, 702),
    L("c12", 2, 8, 10, 13, 12, 3, 3, 1, 1, 703), L("c20", 2, 8, 9, 13, 20, 3, 3, 1, 1, 704), L("c33", 2, 16, 7, 7, 33, 3, 3, 1, 1, 705),
    L("c63", 3, 8, 12, 12, 63, 3, 3, 1, 1, 706), L("c74", 2, 24, 11, 9, 74, 3, 3, 2, 1, 707), L("c95", 2, 8, 8, 31, 95, 3, 3, 1, 1, 708),
    L("c24", 2, 8, 9, 11, 24, 3, 3, 1, 1, 715), L("c40", 2, 16, 10, 9, 40, 3, 3, 2, 1, 716), L("c104", 2, 8, 9, 9, 104, 3, 3, 1, 1, 717),   # whole vectors
    L("c163", 3, 8, 13, 17, 163, 3, 3, 1, 1, 709), L("c301", 2, 16, 9, 9, 301, 3, 3, 1, 1, 710),
    L("parts", 1, 8, 4, 201, 37, 3, 3, 1, 1, 711),          # strips wider than a tile
    L("rounds", 40, 8, 24, 24, 99, 3, 3, 1, 1, 712)], ids=lambda l: l.name)     # more tiles than CTAs
def test_rows_of_any_number_of_channels(layer, kernel, monkeypatch):
    monkeypatch.setenv("IM2WIN_NHWC_KERNEL", kernel)
    dims = layer.dims()
    x, f = workloads.make_small_integer_inputs(layer)
    yr, _ = oracle.conv_direct(x.numpy(), f.numpy(), dims)
    bias = np.arange(layer.Co) % 7 - 3.0
    want = yr.transpose(0, 2, 3, 1)
    for out16 in (False, True):
        assert np.array_equal(gpu_conv_nhwc(x, f, dims, out16=out16, y_nhwc=True), want.astype(np.float16) if out16 else want)
        got = gpu_conv_nhwc(x, f, dims, bias=bias, relu=True, out16=out16, y_nhwc=True)
        ref = np.maximum(want + bias, 0.0)
        assert np.array_equal(got, ref.astype(np.float16) if out16 else ref)


# Rows that meet other CTAs: 78 tile items on 74 CTA pairs, with a reduction long enough that the four tiles of the last round are shared
# between CTAs.  Overlapping rows (98 k-blocks): runs of the reduction, whose partial sums the storing CTA adds up, or halves of the
# channels; shifted views (32 k2-blocks x 3 kernel columns, streamed): K parts, of which the first stores its rows and the others add to
# them (fp32 outputs without ReLU), or quarters of the channels.
SHORT_LAST_ROUND = {"overlap": L("last_overlap", 13, 128, 24, 26, 301, 7, 7, 1, 3, 713), "shift": L("last_shift", 13, 285, 28, 30, 301, 7, 3, 1, 1, 714)}


@functools.lru_cache(maxsize=None)
def short_last_round(kernel):
    layer = SHORT_LAST_ROUND[kernel]
    x, f = workloads.make_small_integer_inputs(layer)
    yr, _ = oracle.conv_direct(x.numpy(), f.numpy(), layer.dims())
    return x, f, yr.transpose(0, 2, 3, 1)


@pytest.mark.parametrize("kernel,switches", [
    ("overlap", {}), ("overlap", {"IM2WIN_NHWC_STREAM": "0"}), ("overlap", {"IM2WIN_NHWC_TAIL": "0"}),
    ("shift", {}), ("shift", {"IM2WIN_NHWC_TAIL_K": "0"}), ("shift", {"IM2WIN_NHWC_TAIL": "0"})],
    ids=["runs", "halves", "overlap_whole", "k_parts", "channel_parts", "shift_whole"])
def test_rows_of_a_short_last_round(kernel, switches, monkeypatch):
    monkeypatch.setenv("IM2WIN_NHWC_KERNEL", kernel)
    monkeypatch.setenv("IM2WIN_NHWC_KSPLIT", "1")
    for k, v in switches.items():
        monkeypatch.setenv(k, v)
    x, f, want = short_last_round(kernel)
    dims = SHORT_LAST_ROUND[kernel].dims()
    bias = np.arange(dims["Co"]) % 7 - 3.0
    assert np.abs(want).max() + 3 < 2048                     # (whole numbers that binary16 holds)
    for out16 in (False, True):
        assert np.array_equal(gpu_conv_nhwc(x, f, dims, out16=out16, y_nhwc=True, packed=True, repeat=3), want)
        assert np.array_equal(gpu_conv_nhwc(x, f, dims, bias=bias, out16=out16, y_nhwc=True), want + bias)
        assert np.array_equal(gpu_conv_nhwc(x, f, dims, bias=bias, relu=True, out16=out16, y_nhwc=True), np.maximum(want + bias, 0.0))


# the transform's strips side by side in a block: short ones, a last block that is not full, channels by 8, 4, 2 and 1
@pytest.mark.parametrize("threads", ["32", "64", "256"])
@pytest.mark.parametrize("layer", [
    L("t3", 3, 3, 9, 11, 8, 3, 3, 1, 1, 720), L("t8", 5, 8, 7, 14, 8, 3, 5, 1, 1, 721), L("t7", 2, 7, 13, 9, 8, 5, 3, 2, 2, 722),
    L("t12", 3, 12, 9, 7, 8, 3, 3, 1, 1, 723), L("t18", 3, 18, 9, 8, 8, 3, 3, 2, 0, 724), L("t35", 2, 35, 11, 13, 8, 1, 1, 2, 0, 725),
    L("t64", 3, 64, 5, 5, 8, 3, 3, 1, 1, 726)], ids=lambda l: l.name)
@pytest.mark.parametrize("layout", ["nchw", "nhwc"])
def test_short_strips_side_by_side(layer, layout, threads, monkeypatch):
    monkeypatch.setenv("IM2WIN_NHWC_STRIP_THREADS", threads)
    dims = layer.dims()
    x, f = workloads.make_small_integer_inputs(layer)
    yr, _ = oracle.conv_direct(x.numpy(), f.numpy(), dims)
    assert np.array_equal(gpu_conv_nhwc(x, f, dims, x_layout=layout), yr)


# tiles whose reduction the CTAs of a cluster share: parts that the k-blocks do not divide into, more CTAs than channels in a tile, several
# channel tiles, tiles of parts of strips, every epilogue
@pytest.mark.parametrize("layer,bn,ctas", [
    (L("s64", 2, 100, 9, 9, 60, 3, 3, 1, 1, 740), 64, 5), (L("s64_16", 1, 200, 7, 8, 5, 5, 3, 1, 1, 741), 64, 16),
    (L("s128", 2, 72, 13, 11, 200, 3, 3, 2, 1, 742), 128, 3), (L("s256", 1, 130, 12, 9, 300, 3, 3, 1, 0, 743), 256, 7),
    (L("s_parts", 1, 40, 4, 150, 37, 3, 5, 1, 1, 744), 64, 2), (L("s_one_kb", 2, 16, 9, 9, 24, 3, 3, 1, 1, 745), 64, 3)], ids=lambda v: getattr(v, "name", str(v)))
def test_shared_tiles(layer, bn, ctas, monkeypatch):
    monkeypatch.setenv("IM2WIN_NHWC_BN", str(bn))
    monkeypatch.setenv("IM2WIN_NHWC_CTAS", str(ctas))
    dims = layer.dims()
    assert binding.im2win_nhwc_kernel_name(dims) == "f16-nhwc-overlap+clusters"
    x, f = workloads.make_small_integer_inputs(layer)
    yr, _ = oracle.conv_direct(x.numpy(), f.numpy(), dims)
    bias = np.arange(layer.Co) % 7 - 3.0
    for y_nhwc in (False, True):
        want = yr.transpose(0, 2, 3, 1) if y_nhwc else yr
        ref = np.maximum(want + (bias if y_nhwc else bias[:, None, None]), 0.0)
        for out16 in (False, True):
            assert np.array_equal(gpu_conv_nhwc(x, f, dims, out16=out16, y_nhwc=y_nhwc), want.astype(np.float16) if out16 else want)
            got = gpu_conv_nhwc(x, f, dims, bias=bias, relu=True, out16=out16, y_nhwc=y_nhwc)
            assert np.array_equal(got, ref.astype(np.float16) if out16 else ref)
    # real values: the order of the parts is fixed, the sums within the tolerance
    x, f = workloads.make_inputs(layer)
    y = gpu_conv_nhwc(x, f, dims)
    yr, ar = oracle.conv_direct(*oracle_inputs(x, f, "f16"), dims)
    check_conv(y, yr, ar, "f16", layer.name)
    assert np.array_equal(gpu_conv_nhwc(x, f, dims), y)
