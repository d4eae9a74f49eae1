"""Host-side rules of the kernel choice (no GPU): which fp32 kernel a layer takes, and that the scratch a caller was told
to provide serves every smaller batch of the same layer, whatever kernel that one takes."""
import os
import random
import subprocess
import sys

import pytest

from conftest import ROOT
from gpu_helpers import runs_form, split_form
from paper_2608_20725_b200 import binding

LAYERS = [(128, 64, 56, 56, 64, 3, 3, 1, 1), (128, 512, 7, 7, 512, 3, 3, 1, 1), (13, 37, 45, 61, 75, 5, 5, 2, 2),
          (64, 256, 28, 28, 256, 11, 11, 1, 5), (128, 3, 224, 224, 64, 7, 7, 2, 3), (96, 9, 15, 17, 270, 2, 3, 1, 1),
          (8, 512, 14, 14, 90, 11, 11, 4, 5), (160, 5, 8, 224, 17, 3, 3, 2, 0)]


@pytest.mark.parametrize("layer", LAYERS, ids=str)
@pytest.mark.parametrize("dtype", [binding.F32, binding.F16])
def test_scratch_serves_smaller_batches(layer, dtype):
    whole = binding.im2win_workspace_size(binding.make_shape(*layer), dtype)[1]
    for n in range(1, layer[0]):
        assert binding.im2win_workspace_size(binding.make_shape(n, *layer[1:]), dtype)[1] <= whole


# (image, kernel) of layers that a kernel no longer takes at the whole batch (2^31 virtual positions, boxes of a tile) but
# takes at a part of it
PARTS = [(8273, 2, 512, 512, 64, 6, 6, 1, 0), (16000, 1, 512, 512, 16, 1, 1, 1, 0), (8, 8, 13, 28, 1, 7, 3, 2, 0),
         (7, 37, 13, 44, 96, 1, 17, 3, 2), (32, 2, 34, 8, 1, 5, 5, 3, 2)]


@pytest.mark.parametrize("layer", PARTS, ids=str)
@pytest.mark.parametrize("dtype", [binding.F32, binding.F16])
def test_scratch_does_not_depend_on_the_batch(layer, dtype):
    size = lambda n: binding.im2win_workspace_size(binding.make_shape(n, *layer[1:]), dtype)[1]
    assert {size(n) for n in (1, 2, 3, layer[0] // 4, layer[0] // 2, layer[0] - 1)} == {size(layer[0])}


@pytest.mark.parametrize("C,K,want", [(3, 3, "f32-ffma"), (63, 1, "f32-ffma"), (64, 1, "f32-split"), (8, 3, "f32-split"),
                                      (600, 11, "f32-ffma")])       # 27, 63, 64, 72 terms; an offset table too long
def test_f32_kernel_by_length_of_the_reduction(C, K, want):
    assert binding.im2win_conv_kernel_name((2, C, 20, 20, 24, K, K, 1, K // 2), binding.F32) == want


@pytest.mark.parametrize("layer,want", [
    ((128, 256, 28, 28, 512, 3, 3, 2, 1), "f16-runs"), ((13, 37, 45, 61, 75, 5, 5, 2, 2), "f16-runs"),
    ((64, 128, 27, 27, 128, 3, 3, 1, 1), "f16-runs"), ((64, 256, 15, 15, 130, 1, 1, 3, 0), "f16-shift"),
    ((128, 512, 7, 7, 512, 3, 3, 1, 1), "f16-shift"),      # several images in a tile: a copy per image and channel
    ((128, 512, 7, 7, 1024, 1, 1, 1, 0), "f16-shift"),     # one element per column and copy
    ((1, 256, 27, 27, 256, 3, 3, 1, 1), "f16-shift"),      # few tiles
    ((32, 64, 61, 45, 64, 3, 3, 1, 0), "f16-shift"),       # 64 channels
    ((128, 128, 35, 9, 128, 7, 5, 1, 3), "f16-runs"), ((128, 128, 35, 9, 129, 7, 5, 1, 3), "f16-shift"),   # five wide, seven high
    ((64, 128, 35, 19, 129, 5, 5, 1, 2), "f16-runs"), ((8, 128, 35, 19, 129, 5, 5, 1, 2), "f16-shift"),    # ... 380 tiles, 48
    ((2, 256, 53, 7, 262, 11, 11, 3, 5), "f16-runs"), ((1, 256, 24, 9, 256, 5, 11, 3, 2), "f16-shift"),    # four virtual columns
    ((16, 256, 8, 8, 64, 3, 3, 1, 1), "f16-runs"), ((16, 256, 4, 6, 64, 3, 3, 1, 1), "f16-shift")])        # images of a tile: 2.6, 5.1
def test_f16_kernel_on_odd_planes(layer, want):
    assert binding.im2win_conv_kernel_name(layer, binding.F16) == want


@pytest.mark.parametrize("layer,want", [
    ((128, 64, 56, 56, 256, 1, 1, 1, 0), "f32-split"), ((128, 64, 56, 56, 300, 1, 1, 1, 0), "f32-ffma"),
    ((8, 80, 28, 28, 128, 1, 1, 1, 0), "f32-ffma"),        # 80 terms in two k2-blocks
    ((8, 81, 28, 28, 128, 1, 1, 1, 0), "f32-split"),
    ((32, 3, 56, 56, 64, 5, 5, 2, 2), "f32-ffma"),         # 75 terms in two column classes
    ((64, 8, 49, 20, 300, 1, 11, 2, 1), "f32-ffma"),       # 88 terms, half of the multiplied ones are zeros
    ((128, 3, 224, 224, 64, 7, 7, 2, 3), "f32-split")])
def test_f32_kernel_on_short_reductions(layer, want):
    assert binding.im2win_conv_kernel_name(layer, binding.F32) == want


def test_switches_are_fixed_when_the_library_is_loaded():
    """Testing-aid switches set after the library was loaded without IM2WIN_DEBUG change nothing: the library and the
    binding, which then keeps sizes, look at it at the same moment."""
    code = ("import os, sys; sys.path.insert(0, sys.argv[1])\n"
            "from paper_2608_20725_b200 import binding\n"
            "binding.lib()\n"
            "os.environ.update(IM2WIN_DEBUG='1', IM2WIN_F32_KERNEL='ffma')\n"
            "print(binding.im2win_conv_kernel_name((2, 64, 20, 20, 24, 3, 3, 1, 1), binding.F32))\n")
    env = {k: v for k, v in os.environ.items() if not k.startswith("IM2WIN_")}
    out = subprocess.run([sys.executable, "-c", code, ROOT], env=env, capture_output=True, text=True, check=True, timeout=300)
    assert out.stdout.split() == ["f32-split"]


def test_run_staged_slots_keep_to_one_team():
    """The team that takes a fill of a raw slot of the run-staged kernel has taken the fill before it too (it waits by the
    parity of the fills): the number of teams divides the number of slots."""
    rng = random.Random(7)
    log = lambda lo, hi: round(lo * (hi / lo) ** rng.random())
    seen = set()
    layers = [(64, 256, 28, 28, 256, 3, 3, 1, 1), (64, 64, 112, 112, 128, 3, 3, 1, 0), (128, 128, 28, 28, 128, 3, 3, 1, 0),
              (64, 128, 56, 56, 64, 3, 3, 1, 1)]
    for _ in range(20000):
        k, st = rng.choice([1, 2, 3, 3, 3, 4, 5, 7, 11]), rng.choice([1, 1, 1, 2, 2, 3, 4])
        layers.append((log(1, 160), log(1, 600), log(7, 224), log(7, 224), log(1, 600), k,
                       rng.choice([k, k, k, 1, 2, 3, 5]), st, rng.choice([0, k // 2])))
    for layer in layers:
        f = runs_form(layer)
        if f is None:
            continue
        assert f.slots % f.teams == 0 and f.teams in ((1,) if f.mode == 3 else (2, 4)) and f.slots % 2 == 0, (layer, f)
        seen.add((f.mode, f.teams))
    assert {m for m, _ in seen} == {0, 1, 2, 3} and {t for _, t in seen} == {1, 2, 4}


@pytest.mark.parametrize("layer,want", [
    ((64, 256, 28, 28, 256, 5, 5, 1, 2), (256, 1, 4)),      # three rounds of tiles and four: the last in quarters
    ((95, 64, 14, 14, 256, 3, 3, 2, 1), (96, 1, 1)),        # one round: narrow tiles, no pairs of CTAs on wide ones
    ((4, 16, 16, 140, 256, 3, 3, 1, 0), (128, 1, 1)),       # ... and no halves of wide ones
    ((32, 128, 20, 20, 256, 3, 7, 1, 1), (256, 1, 1)),      # one round of wide tiles, not two with the last in halves
    ((4, 8, 47, 47, 372, 5, 5, 1, 2), (128, 1, 1))])        # one k2-block: two rounds of narrow tiles
def test_f32_tiles(layer, want):
    assert split_form(layer) == want
