"""Kernels that may start before the one ahead of them in the stream has ended (launch_early, launch_pack, launch_after_previous, or the launch
attribute itself): every thread waits for that one before anything else that reads what it wrote.  A bounded barrier wait counts: its
slow path takes its limit from the status block, which the filter pack clears, so that a wait that came first could give up on a
word left over from whatever the memory held before, and the pack would then clear the status that says so.

Read from the sources: the outcome of such a wait depends on what happens to be in memory.  No GPU needed."""
import ctypes
import os
import re

import pytest

from paper_2608_20725_b200 import binding, build

EARLY = re.compile(r"launch_early\(|launch_pack<|launch_after_previous\(|cudaLaunchAttributeProgrammaticStreamSerialization")
HEAD = re.compile(r"^(?:__global__ void\b.*|__device__ __forceinline__ void \w+_body\(.*|conv_\w+_kernel\(.*)$", re.M)


def bodies(code):
    """(head, body) of every kernel and of every function that is one in all but its launch."""
    at = 0
    while (m := HEAD.search(code, at)) is not None:
        start = code.index("{", m.start())
        depth, end = 1, start + 1
        while depth:
            depth += {"{": 1, "}": -1}.get(code[end], 0)
            end += 1
        yield code[m.start():start], code[start + 1:end - 1]
        at = end


def kernels_that_wait():
    for path in build.sources():
        code = re.sub(r"//[^\n]*", "", open(path).read())
        if EARLY.search(code):
            for head, body in bodies(code):
                if "mbar_wait" in body or "wait_flag(" in body or "wait_for_previous_kernel()" in body:
                    yield pytest.param(body, id=f"{os.path.basename(path)}:{re.findall(r'(\w+)\s*[(]', head.replace('__launch_bounds__', ''))[-1]}")


@pytest.mark.parametrize("body", list(kernels_that_wait()))
def test_every_thread_waits_first(body):
    at = body.find("wait_for_previous_kernel()")
    assert at >= 0, "no wait for the kernel ahead"
    before = body[:at]
    assert "mbar_wait" not in before and "wait_flag(" not in before, "a bounded wait comes first"
    assert before.count("{") == before.count("}"), "inside a branch or a loop: not every thread comes by"


def test_the_kernels_are_found():
    """The ones that start early and have waits: seven convolutions and seven filter packs."""
    ids = [p.id for p in kernels_that_wait()]
    assert len(ids) == len(set(ids)) == 14, ids


@pytest.mark.parametrize("threads,smem", [(256, 0), (256, 5000), (256, 47000), (256, 190000), (320, 90000)])
def test_early_blocks_are_spread_over_the_sms(threads, smem):
    """An SM (228 KB, 1 KB of them for each block) takes its share of the blocks and no more, or what it took anyway if that is less."""
    fn = binding.lib().im2win_spread_smem
    fn.argtypes, fn.restype = [ctypes.c_int64, ctypes.c_int32, ctypes.c_int64], ctypes.c_int64
    anyway = min(2048 // threads, 228 * 1024 // (smem + 1024))
    for blocks in [1, 2, 74, 147, 148, 149, 296, 297, 443, 444, 592, 740, 741, 888, 1036, 1037, 1184, 1185, 5000]:
        asked = fn(blocks, threads, smem)
        share = (blocks + 147) // 148
        assert smem <= asked <= max(smem, 200 * 1024)
        assert min(2048 // threads, 228 * 1024 // (asked + 1024)) == min(share, anyway)
