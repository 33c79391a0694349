"""Planar engine on a GPU: the operand ring in segments of a channel, exact
chunks decided from each segment's largest sample, and the item and unit
numbering, bit for bit against the int64 oracle (8-bit input), for every tile
shape.

Sizes sit at the edges: K-block counts that leave the last segment short (by
one, by all but one), one segment, many; more channels than ring slots; row
counts that fill the last block by one row, or all but one; loud and quiet
stretches of time in turn, so that chunks end inside and at the ends of
segments.
"""
import numpy as np
import pytest
import torch

import oracle
from paper_1107_4264_gb300 import build as engine_build
from paper_1107_4264_gb300 import synth, xc

pytestmark = pytest.mark.gpu

# (N, P, F, T, loudness): loudness "flat" is +-9; "turns" alternates stretches
# of 192 quiet and 192 full-scale samples; "edge" is full scale from the last
# K-block of the first segment on.
CASES = [
    (65, 1, 3, 64, "flat"),       # one K-block; 65 rows of a block
    (129, 1, 2, 576, "turns"),    # nine K-blocks: segments of 5 and 4
    (64, 2, 40, 513, "flat"),     # nine K-blocks, last one with one sample
    (100, 2, 5, 1088, "turns"),   # 17 K-blocks: 6, 6, 5
    (127, 2, 3, 2112, "edge"),    # 33 K-blocks: five segments, 254 rows
    (33, 2, 700, 70, "flat"),     # many channels of one short segment
    (128, 1, 90, 2048, "flat"),   # 360 segments of 512 KiB: the ring goes round
    (200, 2, 9, 1000, "turns"),   # four block rows, the last of 16 inputs
]
SHAPES = [("128", xc.XC_TILE_128), ("pair", xc.XC_TILE_PAIR), ("wide", xc.XC_TILE_WIDE)]


@pytest.fixture(scope="module")
def dev():
    engine_build.build()
    xc.load()
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    return torch.device("cuda:0")


def samples(N, P, F, T, loud, seed):
    x = synth.uniform_int8((T, F, N, P, 2), -9, 9, seed)
    full = synth.uniform_int8((T, F, N, P, 2), -128, 127, seed + 1)
    t = torch.arange(T)
    if loud == "turns":
        x[(t // 192) % 2 == 1] = full[(t // 192) % 2 == 1]
    elif loud == "edge":
        x[448:] = full[448:]
    return x


@pytest.mark.parametrize("N,P,F,T,loud", CASES, ids=["N%d_P%d_F%d_T%d_%s" % c for c in CASES])
def test_segments_bit_exact(N, P, F, T, loud, dev):
    x = samples(N, P, F, T, loud, 3100 + N + T)
    chans = sorted(set([0, 1 % F, F // 2, F - 1]))
    want = oracle.correlate_i8(x[:, chans].contiguous().numpy())
    xd = x.to(dev)
    for name, tile in SHAPES:
        eng = xc.Correlator(N, P, F, T, "int8", tile=tile)
        try:
            for _ in range(2):
                got = eng.correlate(xd, sync=True)
        finally:
            eng.close()
        assert np.array_equal(got[chans].cpu().numpy().astype(np.int64), want), name
