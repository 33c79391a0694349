"""Power-of-two operand scales of float input on a GPU.

Forward: the scale pre-pass must see every sample of every input, whatever the
row length does to its vector loads (odd, even, a multiple of four, shorter and
longer than a block) and wherever the range's remainders fall.  Each input is
small noise with one sample 1e6 times larger at a place of its own, the last
sample and the first among them; a maximum that missed it would overflow fp16.

Adjoint: its operands are scaled per row (input of H, sample of x), so samples
of very different size in one channel each keep their own 22 bits.  Row counts
sit at the kernel's edges: one chunk per thread and four (n = 128, 129), the
widest row kept in registers and one wider (n = 512, 516), and tiles filled by
one sample or all but one.

Tolerances: fp16 operands round each factor within 2^-11, so a product of two
spikes is within 2^-10 (2e-3 leaves room for the noise); hi/lo operands 2e-5,
the bound of the adjoint's other tests, here row by row.
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


@pytest.mark.parametrize("dtype", ["float16", "float32"])
@pytest.mark.parametrize("N,P,F,T", [(1, 1, 2, 1), (3, 1, 7, 65), (5, 2, 3, 513), (65, 1, 2, 129),
                                     (66, 2, 3, 64), (131, 2, 1, 71), (130, 2, 2, 8)])
def test_prepass_sees_every_sample(N, P, F, T, dtype, dev):
    rng = np.random.default_rng(41 + N + T)
    x = (rng.standard_normal((T, F, N, P, 2)) * 1e-3).astype(np.float32)
    n = N * P
    where = (np.arange(F * n) * 37 + T - 1).reshape(F, N, P) % T
    for f in range(F):
        for s in range(N):
            for p in range(P):
                x[where[f, s, p], f, s, p, (s + p) % 2] = 1e3
    x = torch.from_numpy(x).to(getattr(torch, dtype))
    want = oracle.correlate_f64(x.double().numpy())
    eng = xc.Correlator(N, P, F, T, dtype)
    try:
        got = eng.correlate(x.to(dev), sync=True).cpu().double().numpy()
    finally:
        eng.close()
    assert np.isfinite(got).all()
    assert np.abs(got - want).max() <= 2e-3 * 1e6


@pytest.mark.parametrize("N,P,F,T", [(16, 1, 2, 129), (64, 2, 1, 127), (129, 1, 2, 33), (256, 2, 1, 17),
                                     (258, 2, 1, 16), (11, 2, 3, 1)])
def test_adjoint_rows_keep_their_own_scale(N, P, F, T, dev):
    rng = np.random.default_rng(43 + N + T)
    size = 10.0 ** rng.integers(-6, 7, (T, 1, 1, 1, 1))
    x = (rng.standard_normal((T, F, N, P, 2)) * size).astype(np.float32)
    go = rng.standard_normal((F, N * (N + 1) // 2, P * P, 2)).astype(np.float32)
    g = synth.complex_gains(N, P, 43).astype(np.float32)
    gx_want, _ = oracle.backward_f64(x.astype(np.float64), go.astype(np.float64), gains=g.astype(np.float64))
    eng = xc.Correlator(N, P, F, T, "float32")
    try:
        eng.set_gains(torch.from_numpy(g).to(dev))
        gx = eng.correlate_backward(torch.from_numpy(go).to(dev), torch.from_numpy(x).to(dev))
        eng.synchronize()
        gx = gx.cpu().double().numpy()
    finally:
        eng.close()
    err = np.linalg.norm((gx - gx_want).reshape(T, F, -1), axis=-1)
    assert (err <= 2e-5 * np.linalg.norm(gx_want.reshape(T, F, -1), axis=-1)).all()
