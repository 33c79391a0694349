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


# Rows that TMA cannot stride: odd and even numbers of inputs, a half block
# filled by one input or all but one, the last K-block by one sample; fp16 and
# e4m3 operands; few units (dealt one by one) and many (in runs of two).
@pytest.mark.parametrize("precision", [xc.XC_PREC_FP16, xc.XC_PREC_FP8], ids=["fp16", "fp8"])
@pytest.mark.parametrize("N,P,F,T", [(1, 1, 1, 1), (65, 1, 3, 65), (63, 1, 40, 127), (33, 2, 7, 129),
                                     (129, 1, 60, 513), (37, 2, 300, 320)])
def test_unaligned_rows_bit_exact(N, P, F, T, precision, dev):
    x = samples(N, P, F, T, "flat", 3300 + N + T)
    chans = sorted(set([0, F // 2, F - 1]))
    want = oracle.correlate_i8(x[:, chans].contiguous().numpy())
    eng = xc.Correlator(N, P, F, T, "int8", precision=precision, tile=xc.XC_TILE_128)
    try:
        got = eng.correlate(x.to(dev), sync=True)
    finally:
        eng.close()
    assert np.array_equal(got[chans].cpu().numpy().astype(np.int64), want)


@pytest.mark.parametrize("N,P,F,T", [(449, 2, 3, 4033), (448, 2, 2, 4096), (897, 1, 2, 4032)])
def test_default_shape_agrees_with_128(N, P, F, T, dev):
    """Both sides of the rule that picks 128 x 256 items (N P > 896, T > 4032)."""
    x = synth.uniform_int8((T, F, N, P, 2), -9, 9, 3400 + N, device=dev)
    out = []
    for tile in (xc.XC_TILE_AUTO, xc.XC_TILE_128):
        eng = xc.Correlator(N, P, F, T, "int8", tile=tile)
        try:
            out.append(eng.correlate(x, sync=True))
        finally:
            eng.close()
    assert torch.equal(out[0], out[1])
