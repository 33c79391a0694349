"""Hi/lo operands on a GPU with so long an integration that the ring has more
slots than its nominal cap (1172 segments of one channel), on a handle that was
made for fp16 operands, against the FP64 oracle."""
import numpy as np
import pytest
import torch

import oracle
from paper_1107_4264_gb300 import build as engine_build
from paper_1107_4264_gb300 import synth, xc

pytestmark = pytest.mark.gpu


def test_hilo_ring_of_many_segments():
    engine_build.build()
    xc.load()
    N, P, F, T = 2, 1, 2, 300000
    x = synth.sky_voltages(T, F, N, P, noise_sigma=0.7, nsrc=2, src_amp=1.0, seed=3900)
    want = oracle.correlate_f64(x.double().numpy())
    eng = xc.Correlator(N, P, F, T, "float32")
    try:
        before = eng.correlate(x.cuda(), sync=True).cpu().double().numpy()
        eng.set_option(xc.XC_OPT_PRECISION, xc.XC_PREC_HILO)
        for _ in range(2):
            got = eng.correlate(x.cuda(), sync=True).cpu().double().numpy()
    finally:
        eng.close()
    assert np.isfinite(before).all()
    # Operands within 2^-21 per product.  Sums: an MMA adds 16 samples and
    # truncates, 2^-23 of the sum, 12 times per block of 64 samples (three
    # products of four), and the 4688 blocks are rounded, 2^-24 each, into a
    # running sum.
    scale = np.abs(want).max()
    assert np.abs(got - want).max() <= (2.0 ** -21 + 12 * 2.0 ** -23 + 4688 * 2.0 ** -24) * scale
