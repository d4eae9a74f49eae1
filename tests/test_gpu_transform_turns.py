"""Strips and columns per CTA of the NCHW transform: whole turns of a CTA's thread groups, rounded up and down, a last turn nearly full, the most
turns a CTA takes, tensors of few strips or columns; a ragged last CTA, rows that start on odd elements.  Bit for bit against the oracle.
"""
import numpy as np
import pytest
import torch

import oracle
from gpu_helpers import gpu_transform

pytestmark = pytest.mark.gpu


def D(N, C, H, W, Kh, Kw, s, p):
    return dict(N=N, C=C, H=H, W=W, Co=1, Kh=Kh, Kw=Kw, stride=s, pad=p)


@pytest.mark.parametrize("bits", [16, 32])
@pytest.mark.parametrize("dims", [
    D(8, 65, 56, 56, 3, 3, 1, 1),          # fp32: one turn of 32 strips instead of 47; fp16: one of 64, not two
    D(33, 64, 56, 56, 3, 3, 1, 1),         # fp16: two turns of 64 instead of 141
    D(2, 37, 200, 200, 3, 3, 1, 1),        # fp32: rounded up from 13 to 16
    D(4, 30, 224, 224, 7, 7, 2, 3),        # fp16: 15 of 16 stay
    D(4, 51, 145, 145, 1, 1, 1, 0),        # eight turns instead of fourteen
    D(1, 247, 50, 83, 3, 3, 1, 1),         # five turns, odd rows
    D(2, 32, 39, 39, 3, 3, 2, 1), D(3, 3, 7, 5, 1, 1, 1, 0), D(1, 1, 3, 3, 3, 3, 1, 0), D(5, 7, 9, 11, 5, 3, 2, 2),     # few strips
    D(2, 3, 9, 9, 4, 4, 1, 1), D(1, 5, 13, 13, 7, 7, 1, 3), D(7, 40, 61, 61, 2, 2, 1, 0), D(3, 64, 33, 33, 11, 11, 1, 5)],   # columns
    ids=lambda d: f"{d['N']}x{d['C']}x{d['H']}x{d['W']}k{d['Kh']}s{d['stride']}")
def test_transform_turns(dims, bits):
    shape = (dims["N"], dims["C"], dims["H"], dims["W"])
    g = torch.Generator().manual_seed(dims["W"] + bits)
    lim = 2 ** (bits - 1)
    raw = torch.randint(-lim, lim - 1, shape, generator=g, dtype=torch.int64).to(torch.int32 if bits == 32 else torch.int16)
    assert np.array_equal(gpu_transform(raw, dims), oracle.transform(raw.numpy(), dims))
