"""Registers of the planar engine's 8-bit kernels for input that TMA can stride
(the headline path): no spills, in any tile shape, operand format or batch form.
Each converter form needs most of the registers a warp has, so a second one
inlined beside it spills in code that never runs it."""
import os
import re

import pytest

from paper_1107_4264_gb300 import build as engine_build


@pytest.mark.parametrize("src", ["xc_planar.cu", "xc_planar_pair.cu", "xc_planar_wide.cu"])
def test_tma_kernels_do_not_spill(src):
    engine_build.build()
    if not os.path.exists(engine_build.ptxas_log(src)):
        engine_build.build(force=True)
    with open(engine_build.ptxas_log(src)) as fh:
        text = fh.read()
    # planar_*kernel<IS_INT = true, ...>, mangled.
    found = re.findall(r"Compiling entry function '\S*planar_(?:\w+_)?kernelILb1E\S*'.*?(\d+) bytes spill stores, "
                       r"(\d+) bytes spill loads", text, flags=re.S)
    assert len(found) == 3, len(found)  # fp16, fp16 of a batch, e4m3
    assert all(v == ("0", "0") for v in found), found
