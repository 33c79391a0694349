"""CPU check of the planar engine's workspace sizes (xc_planar_plan.h): whatever
operand format a handle is switched to, its ring counters serve that format's
ring, up to the longest integration that is accepted; and a ring always holds a
whole channel's segments."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1107_4264_gb300", "csrc")

HARNESS = r"""
#include <cstdio>
#include "xc_planar_plan.h"
using namespace xc;
int main() {
  const int Ns[] = {1, 2, 64, 65, 256, 1024}, Fs[] = {1, 2, 7, 64, 1024, 65535};
  const int Ts[] = {1, 64, 65, 1000, 8192, 66572, 261120, 262145, 300000, 1000000, 4194240};
  for (int N : Ns) for (int P = 1; P <= 2; ++P) for (int F : Fs) for (int T : Ts) for (int dt = 0; dt < 3; ++dt) {
    if (dt == 0 && T > XC_CI8_MAX_NTIME) continue;
    Geometry g;
    g.N = N; g.P = P; g.F = F; g.T = T;
    g.R = 2 * N * P; g.Tp = (T + 63) / 64 * 64; g.NB = (int64_t)N * (N + 1) / 2;
    const Geometry v = planar_geometry(g, nullptr);
    const int room = planar_max_slots(v, dt, 152);
    const PlanarRing base = planar_ring(v, dt, XC_PREC_FP16, 152);
    for (int fmt = 0; fmt < 3; ++fmt) {
      if (dt == 0 && fmt == XC_PREC_HILO) continue;
      const PlanarRing r = planar_ring(v, dt, fmt, 152);
      std::printf("%d %d %d %d %d %d  %d %d %d %d %d\n", N, P, F, T, dt, fmt, room, r.slots, r.nseg, r.seg_kb, base.nseg);
    }
  }
  return 0;
}
"""


def test_counters_serve_every_format(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not available")
    (tmp_path / "plan.cpp").write_text(HARNESS)
    exe = str(tmp_path / "plan")
    subprocess.run([gxx, "-std=c++17", "-O1", "-I", CSRC, "-I", os.path.join(ROOT, "include"),
                    str(tmp_path / "plan.cpp"), "-o", exe], check=True)
    rows = [[int(v) for v in line.split()]
            for line in subprocess.run([exe], check=True, capture_output=True, text=True).stdout.splitlines()]
    beyond = 0
    for N, P, F, T, dt, fmt, room, slots, nseg, seg_kb, base_nseg in rows:
        what = (N, P, F, T, dt, fmt)
        assert nseg <= slots <= room, what
        assert (nseg - 1) * seg_kb < (T + 63) // 64 <= nseg * seg_kb, what
        if dt == 0:  # the per-segment maxima are sized for fp16 operands
            assert nseg == base_nseg, what
        beyond += slots > 1024
    assert beyond  # rings above the nominal cap are among them
