"""CPU check of the tcgen05 MMA sequences in the kernel sources.

PTX orders back-to-back tcgen05.mma on an accumulator only when they have the
same shape; MMAs of another shape on the same columns may overlap them.  So
all MMAs of a kernel's step loop that add into a pair of accumulators
(d_re, d_im, which lie side by side in TMEM) must take their M and N from one
shape, whatever other bits (negate-B) their descriptors differ in.
"""
import os
import re

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1107_4264_gb300", "csrc")


def shapes(text):
    """Descriptor name -> its "M, N" expression, through "name | flag" definitions."""
    of = dict(re.findall(r"\b(k?[Ii]desc\w*) = (?:ta == 0 \? idesc : )?ptx::idesc_f16_f32\((.*)\);", text))
    for name, base in re.findall(r"\b(k?[Ii]desc\w*) = (k?[Ii]desc\w*) \|", text):
        of[name] = of[base]
    return of


@pytest.mark.parametrize("src", ["xc_planar_kernel.cuh", "xc_adjoint_tc.cu", "xc_small.cu"])
def test_one_shape_per_accumulator_pair(src):
    with open(os.path.join(CSRC, src)) as fh:
        text = fh.read()
    of = shapes(text)
    found = re.findall(r"ptx::mma_f(?:16|8)_ss(?:_pair)?\((\w+), \w+, \w+, (\w+),", text)
    assert found
    used = {}
    for acc, desc in found:
        used.setdefault("pair" if acc in ("d_re", "d_im") else acc, set()).add(of[desc])
    for acc, got in used.items():
        assert len(got) == 1, (src, acc, got)
