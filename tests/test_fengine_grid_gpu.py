"""F-engine on a GPU with more input groups than a second grid dimension could
hold (8-bit output of 512 channels: 16 inputs to a CTA, 65538 of them), against
64-bit DFTs of a few streams at the ends and around the 65536th group."""
import numpy as np
import pytest
import torch

from paper_1107_4264_gb300 import build as engine_build
from paper_1107_4264_gb300 import synth, xc

pytestmark = pytest.mark.gpu


def test_more_than_65535_input_groups():
    engine_build.build()
    xc.load()
    F, P, N = 512, 2, 524304
    x = synth.uniform_int8((N, P, F, 2), -128, 127, 4000, device=torch.device("cuda:0"))
    scale = 0.02
    got = xc.channelize(x, F, scale, "int8")
    torch.cuda.synchronize()
    some = [0, 1, 7, 8, 524279, 524280, 524288, 524303]
    v = x[some].cpu().double().numpy()
    want = np.fft.fft(v[..., 0] + 1j * v[..., 1], axis=-1) * scale  # [stations][P][F]
    code = got[0][:, some].cpu().numpy().transpose(1, 2, 0, 3)      # [stations][P][F][2]
    # Nearest integer of a transform in fp32: 9 levels of butterflies, values up
    # to 128 sqrt(2) 512 scale: 9 * 2^-23 of 1854 is 0.002.
    for part, w in ((code[..., 0], want.real), (code[..., 1], want.imag)):
        assert np.abs(part - np.clip(w, -127, 127)).max() <= 0.5 + 0.002
