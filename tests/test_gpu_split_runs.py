"""The fp32 kernel that runs on the tensor cores (three bf16 pieces per operand) and the run-staged fp16 kernel,
forced over the forms and sizes where they can go wrong: every channel-tile form, tiles shared by clusters of CTAs,
partly filled tiles, k2-blocks and columns, strides that do not divide the strip, several images in a tile, values
that the split cannot hold.

Tolerances: fp32 outputs within 1e-5 * sum|x||w| (gpu_helpers), integer-valued inputs exactly; the error of the split
against the oracle's 64-bit values is at most that of the FFMA kernel on the same inputs.
"""
import numpy as np
import pytest
import torch

import oracle
from paper_2608_20725_b200 import binding, workloads
from paper_2608_20725_b200.workloads import Layer
from gpu_helpers import check_conv, gpu_conv, oracle_inputs

pytestmark = pytest.mark.gpu


def L(name, N, C, H, W, Co, Kh, Kw, s, p, seed, xd="normal01"):
    return Layer(name, N, C, H, W, Co, Kh, Kw, s, p, seed, xd, "he_normal")


# (layer, channel tiles, CTAs per tile) that the plan accepts for it; None: what the library picks
SPLIT = [
    (L("k72", 2, 8, 10, 12, 7, 3, 3, 1, 1, 200), [None, (16, 1)]),                    # shortest reductions, 7 of 16 channels
    (L("co80", 2, 24, 13, 12, 80, 3, 3, 1, 1, 201), [(80, 1), (80, 2), (48, 2), (16, 1)]),   # pieces side by side, two k2-blocks
    (L("co100", 3, 22, 12, 15, 100, 3, 3, 1, 1, 202), [(112, 1), (112, 2), (64, 2)]),   # pieces one by one, the last k2-block one step
    (L("co300", 1, 70, 9, 9, 300, 3, 3, 1, 1, 203), [None, (160, 1), (160, 4), (112, 2), (80, 4), (48, 1)]),
    (L("co256_s2", 2, 33, 15, 17, 256, 3, 3, 2, 1, 204), [(256, 1), (256, 4), (128, 2), (64, 4)]),   # two column classes
    (L("s4_rag", 1, 6, 30, 41, 20, 11, 11, 4, 0, 205), [None, (32, 4), (32, 8)]),     # stride 4, cut-short last column, 2 rows below
    (L("k11", 1, 7, 20, 18, 33, 11, 11, 1, 5, 206), [None, (48, 2)]),                 # ten rows below the tile
    (L("imgs", 9, 30, 5, 5, 40, 3, 3, 1, 1, 207, "uniform01"), [None, (48, 2)]),      # several images in a tile
    (L("k1x1", 3, 130, 7, 7, 65, 1, 1, 1, 0, 208, "uniform01"), [None, (80, 2), (48, 1)]),
    (L("rect", 2, 9, 21, 14, 18, 5, 3, 2, 2, 209), [None, (32, 2)]),
    (L("many_tiles", 40, 16, 24, 24, 24, 3, 3, 1, 1, 210, "uniform01"), [None]),      # more tiles than SMs: the rings go round
]


def force_split(monkeypatch, form):
    monkeypatch.setenv("IM2WIN_F32_KERNEL", "split")
    if form:
        monkeypatch.setenv("IM2WIN_F32_SPLIT_BN", str(form[0]))
        monkeypatch.setenv("IM2WIN_F32_SPLIT_CTAS", str(form[1]))


@pytest.mark.parametrize("layer,form", [(l, f) for l, forms in SPLIT for f in forms], ids=lambda v: getattr(v, "name", str(v)))
def test_conv_f32_split_forms(layer, form, monkeypatch):
    force_split(monkeypatch, form)
    dims = layer.dims()
    assert binding.im2win_conv_kernel_name(dims, binding.F32) == "f32-split"
    x, f = workloads.make_small_integer_inputs(layer)
    y, _, _ = gpu_conv(x, f, dims, "f32")
    yr, _ = oracle.conv_direct(x.numpy(), f.numpy(), dims)
    assert np.array_equal(y.astype(np.float64), yr)
    x, f = workloads.make_inputs(layer)
    y, _, _ = gpu_conv(x, f, dims, "f32")
    yr, ar = oracle.conv_direct(x.numpy(), f.numpy(), dims)
    check_conv(y, yr, ar, "f32", layer.name)
    monkeypatch.setenv("IM2WIN_F32_KERNEL", "ffma")
    z, _, _ = gpu_conv(x, f, dims, "f32")
    assert np.linalg.norm(y - yr) <= np.linalg.norm(z - yr)


@pytest.mark.parametrize("form", [(80, 1), (80, 2), (112, 1), (256, 2)], ids=str)
@pytest.mark.parametrize("what", ["inf", "nan", "lowest", "overflow", "inf weight", "tiny", "subnormal", "tiny weight"])
def test_conv_f32_split_values_beyond_the_pieces(form, what, monkeypatch):
    """Outputs that meet infinities, NaNs, values next to the largest finite one, or only values so small that pieces
    are lost, are what the FFMA kernel computes: the same bits where they are not finite or tiny, and nothing else is
    disturbed."""
    layer = L("values", 2, 24, 9, 12, form[0] - 5, 3, 3, 1, 1, 220)
    dims = layer.dims()
    x, f = workloads.make_inputs(layer)
    x, f = x.clone(), f.clone()
    if what == "inf": x[0, 3, 4, 5] = float("inf")
    if what == "nan": x[1, 7, 0, 11] = float("nan")
    if what == "lowest": x[0, 1] = torch.finfo(torch.float32).min
    if what == "overflow":                   # (one sign, so that no order of the sum stays finite)
        x[1, :, 2] = 3e38
        f = f.abs()
    if what == "inf weight": f[6, 2, 1, 1] = float("-inf")
    if what == "tiny": x *= 1e-36
    if what == "subnormal": x *= 1e-39
    if what == "tiny weight": f *= 1e-37
    force_split(monkeypatch, form)
    y, _, _ = gpu_conv(x, f, dims, "f32")
    monkeypatch.setenv("IM2WIN_F32_KERNEL", "ffma")
    z, _, _ = gpu_conv(x, f, dims, "f32")
    same = (y == z) | (np.isnan(y) & np.isnan(z))
    odd = ~np.isfinite(z) | (np.abs(z) < 2.0 ** -90)
    assert odd.any() or what == "lowest"
    assert same[odd].all() and np.array_equal(np.isfinite(y), np.isfinite(z))
    ok = ~odd
    if ok.any():
        a, b = y[ok].astype(np.float64), z[ok].astype(np.float64)
        scale = np.abs(b).max()
        assert np.linalg.norm((a - b) / scale) <= 1e-6 * np.linalg.norm(b / scale)


@pytest.mark.parametrize("co", [16, 33, 64, 80])
def test_conv_f32_split_starts_from_clean_accumulators(co, monkeypatch):
    """No output depends on what tensor memory held before: with NaNs left in all of its columns on every SM, a layer of
    many tiles gives the same bits again and again, and the oracle's values."""
    left = L("left", 40, 8, 24, 24, 256, 3, 3, 1, 1, 211)
    layer = L("clean", 40, 40, 24, 24, co, 3, 3, 1, 1, 212)
    x0, f0 = workloads.make_inputs(left)
    x, f = workloads.make_inputs(layer)
    yr, ar = oracle.conv_direct(x.numpy(), f.numpy(), layer.dims())
    first = None
    for _ in range(3):
        force_split(monkeypatch, (256, 1))
        gpu_conv(torch.full_like(x0, float("nan")), f0, left.dims(), "f32")
        force_split(monkeypatch, ((co + 15) // 16 * 16, 1))
        y, _, _ = gpu_conv(x, f, layer.dims(), "f32")
        first = y if first is None else first
        assert np.array_equal(y, first)
    check_conv(first, yr, ar, "f32", layer.name)


@pytest.mark.parametrize("form", [(64, 1), (64, 2), (112, 1), (256, 2)], ids=str)
@pytest.mark.parametrize("xs,fs", [(-100, 30), (-112, 40), (-124, 60), (-137, 60), (-145, 100), (40, -112), (60, -137),
                                   (100, -145), (90, -50), (80, 5), (110, -120)])
def test_conv_f32_split_holds_operands_of_any_size(form, xs, fs, monkeypatch):
    """Small elements on one side and large ones on the other: the outputs are of ordinary size, and as close to the
    64-bit values as the FFMA kernel's, although the operands' low bits lie far below bf16's range."""
    layer = L("sizes", 2, 64, 9, 12, form[0] - 5, 3, 3, 1, 1, 221)
    dims = layer.dims()
    x, f = workloads.make_inputs(layer)
    x, f = (x.double() * 2.0 ** xs).float(), (f.double() * 2.0 ** fs).float()
    yr, ar = oracle.conv_direct(x.numpy(), f.numpy(), dims)
    force_split(monkeypatch, form)
    y, _, _ = gpu_conv(x, f, dims, "f32")
    check_conv(y, yr, ar, "f32", layer.name)
    monkeypatch.setenv("IM2WIN_F32_KERNEL", "ffma")
    z, _, _ = gpu_conv(x, f, dims, "f32")
    scale = 1.0 / np.abs(yr).max()
    assert np.linalg.norm((y - yr) * scale) <= np.linalg.norm((z - yr) * scale)


def device_seconds(call):
    start, stop = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    call()
    start.record()
    call()
    stop.record()
    stop.synchronize()
    return start.elapsed_time(stop) / 1e3


@pytest.mark.parametrize("what", ["nan", "inf", "tiny"])
def test_conv_f32_split_recomputes_whole_tensors_in_bounded_time(what, monkeypatch):
    """Every output of a long reduction computed again: the same values as the FFMA kernel, well inside the time after
    which a device-side wait gives up (4 s), although one CTA has the whole tile.  (One output at a time: 128 x 26112
    dependent steps of some 500 cycles, 0.9 s.)"""
    layer = L("long", 8, 96, 16, 40, 256, 16, 17, 1, 0, 222)
    dims = layer.dims()
    force_split(monkeypatch, (256, 1))
    x, f = workloads.make_inputs(layer)
    x, f = {"nan": (torch.full_like(x, float("nan")), f), "inf": (torch.full_like(x, float("inf")), f),
            "tiny": (x * 1e-30, f * 1e-10)}[what]
    window, scratch, y = binding.alloc_layer_buffers(dims, torch.float32)
    xd, fd = x.cuda(), f.cuda()
    binding.im2win_transform(xd, window, dims)
    binding.im2win_pack_filter(fd, scratch, dims)
    seconds = device_seconds(lambda: binding.im2win_conv_packed(window, y, scratch, dims))
    binding.im2win_check_status(scratch)
    monkeypatch.setenv("IM2WIN_F32_KERNEL", "ffma")
    z, _, _ = gpu_conv(x, f, dims, "f32")
    y = y.cpu().numpy()
    assert ((y == z) | (np.isnan(y) & np.isnan(z))).all()
    assert seconds < 0.25


@pytest.mark.parametrize("precision,layer", [("f32", L("co524289", 1, 64, 4, 4, 524289, 1, 1, 1, 0, 250)),
                                             ("f16", L("co524289", 1, 3, 9, 9, 524289, 3, 3, 2, 1, 251))], ids=["f32", "f16"])
def test_filter_pack_takes_any_number_of_channels(precision, layer, monkeypatch):
    """More channel blocks than the second axis of a grid has (65535)."""
    monkeypatch.setenv("IM2WIN_F16_KERNEL", "runs")
    monkeypatch.setenv("IM2WIN_F32_KERNEL", "split")
    dims = layer.dims()
    code = binding.F32 if precision == "f32" else binding.F16
    assert binding.im2win_conv_kernel_name(dims, code) == ("f32-split" if precision == "f32" else "f16-runs")
    x, f = workloads.make_inputs(layer)
    y, _, _ = gpu_conv(x, f, dims, precision)
    for part in (slice(0, 40), slice(layer.Co - 40, layer.Co)):
        xo, fo = oracle_inputs(x, f[part], precision)
        yr, ar = oracle.conv_direct(xo, fo, dict(dims, Co=40))
        check_conv(y[:, part], yr, ar, precision, layer.name)


@pytest.mark.parametrize("layer", [L("host_tiles", 32, 256, 28, 28, 256, 3, 3, 1, 1, 260),    # the parts alone: other tiles, clusters
                                   L("host_clusters", 40, 72, 28, 28, 64, 3, 3, 1, 1, 261),
                                   L("host_ffma", 24, 7, 70, 70, 64, 3, 3, 1, 1, 262)], ids=lambda l: l.name)
def test_layer_forward_host_in_parts_gives_the_bits_of_the_whole(layer):
    dims = layer.dims()
    x, f = workloads.make_inputs(layer)
    assert (x.numel() + layer.N * layer.Co * layer.H * layer.W) * 4 >= 8 << 20      # large enough to go in four parts
    y, _, _ = gpu_conv(x, f, dims, "f32")
    out = torch.full(y.shape, float("nan")).pin_memory()
    ws = torch.empty(binding.im2win_layer_workspace_size(dims, binding.F32), dtype=torch.uint8, device="cuda")
    binding.im2win_layer_forward_host(x.pin_memory(), f.pin_memory(), out, ws, dims)
    torch.cuda.synchronize()
    assert np.array_equal(out.numpy(), y)


RUNS = [l for l, _ in SPLIT if l.name != "s4_rag"] + [         # (its rings do not fit that one)
    L("runs_s4", 1, 6, 30, 41, 20, 7, 7, 4, 0, 235),         # stride 4, cut-short last column, a row below the tile
    L("runs_quad", 2, 3, 19, 23, 20, 7, 7, 2, 3, 230),       # up to four channels: a unit is four channels at two columns' elements
    L("runs_quad1", 3, 2, 12, 9, 16, 1, 1, 1, 0, 231),       # ... one unit, one step
    L("runs_ragged3", 2, 7, 20, 21, 9, 4, 4, 3, 0, 232),     # stride 3, cut-short last column, tensor ends off a 16-byte boundary
    L("runs_c9", 2, 9, 15, 17, 270, 2, 3, 1, 1, 233),        # an octet with one channel, two channel tiles
    L("runs_resident", 6, 24, 30, 30, 48, 3, 3, 1, 1, 234),  # filter resident, tiles enough to go round the rings
]


@pytest.mark.parametrize("layer", RUNS, ids=lambda l: l.name)
def test_conv_f16_runs(layer, monkeypatch):
    monkeypatch.setenv("IM2WIN_F16_KERNEL", "runs")
    dims = layer.dims()
    assert binding.im2win_conv_kernel_name(dims, binding.F16) == "f16-runs"
    x, f = workloads.make_small_integer_inputs(layer)
    y, _, _ = gpu_conv(x, f, dims, "f16")
    yr, _ = oracle.conv_direct(x.numpy(), f.numpy(), dims)
    assert np.array_equal(y.astype(np.float64), yr)
    x, f = workloads.make_inputs(layer)
    y, _, _ = gpu_conv(x, f, dims, "f16")
    xo, fo = oracle_inputs(x, f, "f16")
    yr, ar = oracle.conv_direct(xo, fo, dims)
    check_conv(y, yr, ar, "f16", layer.name)
    # an infinity and a NaN reach exactly the outputs whose windows hold them (strided kernels are widened by zeros)
    xs = x.clone()
    xs.view(-1)[xs.numel() // 3] = float("inf")
    xs.view(-1)[xs.numel() // 2] = float("nan")
    y, _, _ = gpu_conv(xs, f, dims, "f16")
    monkeypatch.setenv("IM2WIN_F16_KERNEL", "gather")
    z, _, _ = gpu_conv(xs, f, dims, "f16")
    odd = ~np.isfinite(z)
    assert np.array_equal(np.isfinite(y), ~odd) and np.array_equal(np.isnan(y), np.isnan(z))
    assert np.array_equal(np.sign(y[np.isinf(z)]), np.sign(z[np.isinf(z)]))


@pytest.mark.parametrize("layer", [L("down", 4, 256, 28, 28, 512, 3, 3, 2, 1, 240),       # columns beyond the kernel's width
                                   L("c27", 4, 128, 27, 27, 128, 3, 3, 1, 1, 241),        # nothing foreign meets a zero
                                   L("c9", 4, 129, 27, 27, 128, 3, 3, 1, 1, 242)],        # channels beyond the last
                         ids=lambda l: l.name)
@pytest.mark.parametrize("what", ["nan", "inf", "one nan"])
def test_conv_f16_runs_not_finite_tensors_in_bounded_time(layer, what, monkeypatch):
    """Tensors full of NaNs or infinities, and one NaN in a plain tensor: the classes the gather kernel gives.  A plain pass
    takes 0.1 ms and less; one output at a time took 39 ms for a single NaN."""
    dims = layer.dims()
    monkeypatch.setenv("IM2WIN_F16_KERNEL", "runs")
    assert binding.im2win_conv_kernel_name(dims, binding.F16) == "f16-runs"
    x, f = workloads.make_inputs(layer)
    if what == "one nan":
        x = x.clone()
        x[1, 3, 14, 13] = float("nan")
    else:
        x = torch.full_like(x, float(what))
    window, scratch, y = binding.alloc_layer_buffers(dims, torch.float16)
    xd, fd = x.half().cuda(), f.half().cuda()
    binding.im2win_transform(xd, window, dims)
    binding.im2win_pack_filter(fd, scratch, dims)
    seconds = device_seconds(lambda: binding.im2win_conv_packed(window, y, scratch, dims))
    binding.im2win_check_status(scratch)
    z, _, _ = gpu_conv(x, f, dims, "f16-gather")
    y = y.cpu().numpy()
    assert np.array_equal(np.isnan(y), np.isnan(z)) and np.array_equal(np.isinf(y), np.isinf(z))
    assert np.array_equal(np.sign(y[np.isinf(z)]), np.sign(z[np.isinf(z)]))
    assert seconds < 5e-3


DROP_ARRIVE = 0x0d0a11fe      # word 2 of the status block: the first CTA leaves out one arrival (csrc/ptx_sm100.cuh)


@pytest.mark.parametrize("dtype,layer,form", [
    (torch.float32, L("wait_split", 4, 64, 12, 12, 64, 3, 3, 1, 1, 270), (64, 1)),
    (torch.float32, L("wait_wide", 4, 64, 12, 12, 256, 3, 3, 1, 1, 271), (256, 1)),
    (torch.float32, L("wait_cluster", 4, 64, 12, 12, 112, 3, 3, 1, 1, 272), (112, 2)),    # the other CTA of the cluster goes on
    (torch.float16, L("wait_runs", 4, 64, 12, 12, 130, 3, 3, 2, 1, 273), None)], ids=lambda v: getattr(v, "name", None))
def test_a_wait_that_cannot_complete_gives_up_and_the_kernel_returns(dtype, layer, form, monkeypatch):
    """One arrival left out and the poll limit lowered (testing aids of the status block): the kernel returns with the status
    raised, nothing faults or hangs, and the same layer computes as ever afterwards (its tensor memory was given back)."""
    if form:
        force_split(monkeypatch, form)
    else:
        monkeypatch.setenv("IM2WIN_F16_KERNEL", "runs")
    dims = layer.dims()
    precision = "f32" if form else "f16"
    x, f = workloads.make_inputs(layer)
    want, _, _ = gpu_conv(x, f, dims, precision)
    xd, fd = x.to(dtype).cuda(), f.to(dtype).cuda()
    window, scratch, y = binding.alloc_layer_buffers(dims, dtype)
    binding.im2win_transform(xd, window, dims)
    binding.im2win_pack_filter(fd, scratch, dims)
    torch.cuda.synchronize()
    words = scratch[:256].view(torch.int32)
    words[1] = 4096
    words[2] = DROP_ARRIVE
    binding.im2win_conv_packed(window, y, scratch, dims)
    with pytest.raises(binding.Im2winError) as err:
        binding.im2win_check_status(scratch)
    assert err.value.code == 7
    for _ in range(2):
        y.fill_(float("nan"))
        binding.im2win_pack_filter(fd, scratch, dims)
        binding.im2win_conv_packed(window, y, scratch, dims)
        binding.im2win_check_status(scratch)
        assert np.array_equal(y.cpu().numpy(), want)


@pytest.mark.parametrize("precision", ["f32", "f16"])
def test_two_streams(precision, monkeypatch):
    """Passes of two layers on two streams, each with its own buffers, give what each gives alone."""
    monkeypatch.setenv("IM2WIN_F32_KERNEL", "split")
    monkeypatch.setenv("IM2WIN_F16_KERNEL", "runs")
    dtype = torch.float32 if precision == "f32" else torch.float16
    work = []
    for layer in (L("s0", 24, 64, 20, 20, 64, 3, 3, 1, 1, 280), L("s1", 16, 72, 18, 18, 200, 3, 3, 2, 1, 281)):
        x, f = workloads.make_inputs(layer)
        want, _, _ = gpu_conv(x, f, layer.dims(), precision)
        window, scratch, y = binding.alloc_layer_buffers(layer.dims(), dtype)
        work.append((layer.dims(), x.to(dtype).cuda(), f.to(dtype).cuda(), window, scratch, y, want, torch.cuda.Stream()))
    torch.cuda.synchronize()
    for _ in range(20):
        for dims, x, f, window, scratch, y, _, stream in work:
            binding.im2win_transform(x, window, dims, stream)
            (binding.im2win_conv_f32 if precision == "f32" else binding.im2win_conv_f16)(window, f, y, scratch, dims, stream)
    for dims, x, f, window, scratch, y, want, stream in work:
        binding.im2win_check_status(scratch, stream)
        assert np.array_equal(y.cpu().numpy(), want)
