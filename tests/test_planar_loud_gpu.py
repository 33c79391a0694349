"""Planar engine on a GPU: loud 8-bit integrations of several exact chunks, in
channels of which the operand ring holds only a part at a time, bit for bit
against the int64 oracle: every tile shape, one loud channel among quiet ones,
rows that TMA cannot stride, a batch, and the no-allocation call's ring.

A visibility depends on its two stations only, so the oracle takes the stations
at the edges of the 128-input blocks and a few in between.
"""
import numpy as np
import pytest
import torch

import oracle
from paper_1107_4264_gb300 import build as engine_build
from paper_1107_4264_gb300 import synth, xc

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dev():
    engine_build.build()
    xc.load()
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    return torch.device("cuda:0")


def samples(N, P, F, T, loud, seed, dev):
    """Full scale in every channel ("all"), or in channel 5 alone and +-9 elsewhere ("one")."""
    if loud == "all":
        return synth.uniform_int8((T, F, N, P, 2), -128, 127, seed, device=dev)
    x = synth.uniform_int8((T, F, N, P, 2), -9, 9, seed, device=dev)
    x[:, 5] = synth.uniform_int8((T, N, P, 2), -128, 127, seed + 1, device=dev)
    return x


def check(x, got, what):
    T, F, N, P, _ = x.shape
    step = 128 // P
    st = sorted({s for b in range(0, N, step) for s in (b, b + 1, b + step // 2, b + step - 1) if s < N} | {N - 1})
    chans = sorted({0, 5 % F, F // 2, F - 1})
    want = oracle.correlate_i8(x[:, chans][:, :, st].contiguous().cpu().numpy())
    idx = [st[i] * (st[i] + 1) // 2 + st[j] for i in range(len(st)) for j in range(i + 1)]
    assert np.array_equal(got[chans][:, idx].cpu().numpy().astype(np.int64), want), what


SHAPES = [("auto", xc.XC_TILE_AUTO), ("128", xc.XC_TILE_128), ("pair", xc.XC_TILE_PAIR), ("wide", xc.XC_TILE_WIDE)]


@pytest.mark.parametrize("N,P,F,T,loud", [(100, 2, 64, 4096, "all"), (256, 2, 16, 8192, "all"),
                                          (128, 2, 256, 4096, "one"), (512, 2, 16, 8192, "all"),
                                          (73, 1, 300, 4099, "all")])
def test_loud_long_bit_exact(N, P, F, T, loud, dev):
    x = samples(N, P, F, T, loud, 3600 + N, dev)
    for name, tile in SHAPES:
        eng = xc.Correlator(N, P, F, T, "int8", tile=tile)
        try:
            for _ in range(2):
                got = eng.correlate(x, sync=True)
            check(x, got, name)
        finally:
            eng.close()


def test_loud_long_batch(dev):
    subs = [(100, 64, 4096), (256, 16, 8192), (33, 40, 2000)]  # (N, F, T)
    xs = [samples(N, 2, F, T, "all", 3700 + N, dev) for N, F, T in subs]
    for tile in (xc.XC_TILE_AUTO, xc.XC_TILE_PAIR, xc.XC_TILE_WIDE):
        bc = xc.BatchCorrelator(subs, npol=2)
        try:
            bc.set_option(xc.XC_OPT_TILE, tile)
            outs = bc.correlate(xs, sync=True)
            for x, o in zip(xs, outs):
                check(x, o, tile)
        finally:
            bc.close()


def test_loud_long_noalloc(dev):
    N, P, F, T = 256, 2, 16, 8192
    x = samples(N, P, F, T, "all", 3800, dev)
    out = torch.empty((F, N * (N + 1) // 2, P * P, 2), dtype=torch.int32, device=dev)
    status = torch.zeros(1, dtype=torch.int32, device=dev)
    st = xc.xc_correlate_noalloc(N, P, F, T, xc.XC_CI8, x.data_ptr(), out.data_ptr(), status.data_ptr(),
                                 torch.cuda.current_stream(dev).cuda_stream)
    assert st == xc.XC_OK, xc.xc_last_error_message()
    torch.cuda.synchronize(dev)
    assert int(status.item()) == 0
    check(x, out, "noalloc")
