"""Tiles whose reduction the CTAs of a cluster share: every form of the fp32 tensor-core kernel, numbers of CTAs that divide neither the
k-blocks nor the channels, shares without a channel; and which layers are shared.

Tolerances: those of gpu_helpers (the sum of a part is an fp32 accumulator's, and up to 16 of them are added in fp32); integer-valued
inputs exactly.
"""
import numpy as np
import pytest
import torch

import oracle
from paper_2608_20725_b200 import binding, workloads
from paper_2608_20725_b200.workloads import Layer
from gpu_helpers import check_conv, gpu_conv, oracle_inputs, split_form


def L(name, N, C, H, W, Co, Kh, Kw, s, p, seed, xd="normal01"):
    return Layer(name, N, C, H, W, Co, Kh, Kw, s, p, seed, xd, "he_normal")


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


@pytest.mark.parametrize("layer,form", [
    ((2, 256, 35, 35, 78, 7, 7, 1, 0), (48, 4)),     # 16 tiles: only 15 clusters of 8 are resident at once
    ((4, 512, 14, 14, 90, 11, 11, 4, 5), (16, 16)),
    ((1, 256, 8, 8, 103, 3, 3, 1, 0), (16, 12))])
def test_which_fp32_layers_are_shared(layer, form):
    assert split_form(layer)[:2] == form
