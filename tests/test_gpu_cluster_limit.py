"""Clusters that share a tile on a device that cannot hold clusters as wide as the plan's (a MIG slice, an MPS share): the launchers take the
widest that fit, or the unshared form, and every layer still runs.  IM2WIN_CLUSTER_LIMIT stands for such a device.

Integer-valued inputs exactly; real values bit for bit as with that number of CTAs asked for (the parts of a sum are added in rank
order), which also shows that the whole device takes the clusters of the plan.
"""
import ctypes

import numpy as np
import pytest

import oracle
from paper_2608_20725_b200 import binding, workloads
from paper_2608_20725_b200.workloads import Layer
from gpu_helpers import gpu_conv, gpu_conv_nhwc


def L(name, N, C, H, W, Co, Kh, Kw, s, p, seed):
    return Layer(name, N, C, H, W, Co, Kh, Kw, s, p, seed, "normal01", "he_normal")


@pytest.mark.parametrize("resident,want,got", [
    ({z: 7 for z in range(1, 17)}, 16, 16), ({z: 7 for z in range(1, 17)}, 5, 5),
    ({z: 2 for z in range(1, 9)}, 16, 8), ({z: 2 for z in range(1, 9)}, 8, 8), ({z: 2 for z in range(1, 9)}, 3, 3),
    ({1: 4, 2: 2, 4: 1}, 12, 4), ({1: 4, 2: 2, 4: 1}, 3, 2), ({1: 4}, 16, 1), ({}, 7, 1), ({1: 4}, 1, 1)])
def test_widest_cluster_of_a_device(resident, want, got):
    """The rule alone: clusters of z CTAs that the device holds -> CTAs taken for what the plan wants.  No GPU needed."""
    fn = binding.lib().im2win_widest_cluster
    fn.argtypes, fn.restype = [ctypes.c_int32, ctypes.POINTER(ctypes.c_int32)], ctypes.c_int32
    assert fn(want, (ctypes.c_int32 * 17)(*[resident.get(z, 0) for z in range(17)])) == got


KERNELS = {
    "f32": (L("f32", 1, 150, 8, 11, 100, 3, 3, 2, 1, 760), {"IM2WIN_F32_KERNEL": "split", "IM2WIN_F32_SPLIT_BN": "112"}, "IM2WIN_F32_SPLIT_CTAS", 9),
    "runs": (L("runs", 1, 200, 14, 12, 40, 3, 3, 1, 1, 761), {"IM2WIN_F16_KERNEL": "runs"}, "IM2WIN_F16_SPLIT", 9),
    "runs_256": (L("runs_256", 2, 130, 14, 12, 160, 3, 3, 1, 1, 762), {"IM2WIN_F16_KERNEL": "runs"}, "IM2WIN_F16_SPLIT", 6),
    "runs_units": (L("runs_units", 1, 48, 20, 20, 24, 11, 11, 2, 5, 763), {"IM2WIN_F16_KERNEL": "runs"}, "IM2WIN_F16_SPLIT", 12),
    "shift_64": (L("shift_64", 1, 350, 6, 6, 9, 3, 3, 1, 1, 764), {"IM2WIN_F16_KERNEL": "shift", "IM2WIN_F16_SHIFT_BN": "64"}, "IM2WIN_F16_SPLIT", 16),
    "shift_128": (L("shift_128", 2, 100, 17, 13, 70, 3, 3, 2, 1, 765), {"IM2WIN_F16_KERNEL": "shift", "IM2WIN_F16_SHIFT_BN": "128"}, "IM2WIN_F16_SPLIT", 5),
    "shift_256": (L("shift_256", 2, 75, 9, 9, 300, 3, 3, 1, 1, 766), {"IM2WIN_F16_KERNEL": "shift", "IM2WIN_F16_SHIFT_BN": "256"}, "IM2WIN_F16_SPLIT", 4),
}


@pytest.mark.gpu
@pytest.mark.parametrize("limit", [3, 1])
@pytest.mark.parametrize("name", KERNELS)
def test_layers_run_with_the_clusters_that_fit(name, limit, monkeypatch):
    layer, forced, ctas_switch, ctas = KERNELS[name]
    precision = "f32" if name == "f32" else "f16"
    dims = layer.dims()
    for k, v in forced.items():
        monkeypatch.setenv(k, v)

    def run(x, f, ctas, limit=None):
        monkeypatch.setenv(ctas_switch, str(ctas))
        if limit is not None:
            monkeypatch.setenv("IM2WIN_CLUSTER_LIMIT", str(limit))
        y, _, _ = gpu_conv(x, f, dims, precision)
        monkeypatch.delenv("IM2WIN_CLUSTER_LIMIT", raising=False)
        return y

    x, f = workloads.make_small_integer_inputs(layer)
    yr, _ = oracle.conv_direct(x.numpy(), f.numpy(), dims)
    assert np.array_equal(run(x, f, ctas, limit), yr)
    x, f = workloads.make_inputs(layer)
    whole, narrow, asked = run(x, f, ctas), run(x, f, ctas, limit), run(x, f, limit)
    assert np.array_equal(narrow, asked) and not np.array_equal(narrow, whole)
    assert np.array_equal(run(x, f, ctas), whole)              # (nothing of the narrow device is kept)


@pytest.mark.gpu
@pytest.mark.parametrize("limit", [2, 1])
@pytest.mark.parametrize("bn,ctas", [(64, 5), (128, 3), (256, 7)])
def test_nhwc_layers_run_with_the_clusters_that_fit(bn, ctas, limit, monkeypatch):
    layer = L("nhwc", 1, 130, 12, 9, 300, 3, 3, 1, 0, 767)
    dims = layer.dims()
    monkeypatch.setenv("IM2WIN_NHWC_BN", str(bn))
    monkeypatch.setenv("IM2WIN_NHWC_KERNEL", "overlap")
    x, f = workloads.make_small_integer_inputs(layer)
    yr, _ = oracle.conv_direct(x.numpy(), f.numpy(), dims)
    bias = np.arange(layer.Co) % 7 - 3.0
    want = np.maximum(yr + bias[:, None, None], 0.0).astype(np.float16)
    real = workloads.make_inputs(layer)
    alone = gpu_conv_nhwc(*real, dims)
    monkeypatch.setenv("IM2WIN_NHWC_CTAS", str(ctas))
    whole = gpu_conv_nhwc(*real, dims)
    monkeypatch.setenv("IM2WIN_CLUSTER_LIMIT", str(limit))
    assert np.array_equal(gpu_conv_nhwc(x, f, dims), yr)
    assert np.array_equal(gpu_conv_nhwc(x, f, dims, bias=bias, relu=True, out16=True), want)
    narrow = gpu_conv_nhwc(*real, dims)
    monkeypatch.delenv("IM2WIN_CLUSTER_LIMIT")
    monkeypatch.setenv("IM2WIN_NHWC_CTAS", str(limit))
    asked = alone if limit == 1 else gpu_conv_nhwc(*real, dims)
    assert np.array_equal(narrow, asked) and not np.array_equal(narrow, whole)
