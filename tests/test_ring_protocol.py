"""CPU model of the planar engine's operand-ring protocol: can it stall?

Converter warps, and per CTA the producer, the MMA warp and the epilogue, walk
their work as in the kernel (xc_planar_kernel.cuh) and wait on the same
counters, stages and accumulator sets; ring, segments and waves are the ones
xc_planar_plan.h gives the launch.  Every wait is for a count that only grows,
so whatever order the roles are stepped in they end in the same state: all
done, or stuck for good.

The epilogue is modelled in two ways: waiting for full accumulators alone (the
kernel), and waiting for the whole channel to be converted first.  The second
must stall on loud 8-bit input whose channels the ring does not hold: the MMA
warp then waits for a drain of an exact chunk, the epilogue for segments whose
slots only that MMA warp can free.  A model that did not show it would show
nothing about the first.
"""
import os
import random
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1107_4264_gb300", "csrc")

HARNESS = r"""
#include <cstdio>
#include <cstdlib>
#include <vector>
#include "xc_planar_plan.h"
using namespace xc;
typedef long long ll;

struct Sub {
  Geometry g;
  PlanarRing r;
  int nib, nkb, ipc, wave, seg_units, loud;
  std::vector<unsigned> ready, done;
  // Channel f's segments: first, first + width, ...
  int first(int f, int* width) const {
    const int w = f / wave, full = g.F / wave;
    *width = w < full ? wave : g.F - full * wave;
    return w * wave * r.nseg + f - w * wave;
  }
  // Growth of a partial sum per K-block.  loud: max |x|; negative: that in one
  // channel of 16 and 3 in the others; 1000 + s: random per segment.
  unsigned grow(int f, int seg) const {
    unsigned m = loud;
    if (loud < 0) m = f % 16 == 5 ? -loud : 3;
    if (loud >= 1000) {
      const unsigned h = (f * 7919u + seg * 104729u + loud * 31u) * 2654435761u >> 24;
      m = h < 64 ? 128 : h < 128 ? 60 : h < 192 ? 9 : 0;
    }
    return 2 * m * m * 64;
  }
};

struct Warp {
  ll u;
  int claimed_G = -1, claimed_sb = -1;
  Sub* pend = nullptr;  // converted units not yet published
  int pend_slot = 0;
  ll pend_run = -1;
  unsigned pend_n = 0;
  bool fin = false;
};
struct Word { bool start, end; };
struct Group { int sb, f; };
struct Cta {
  // Producer.
  ll it; int kb = 0, st = 0, f_left = 0; unsigned sum = 0; ll issued = 0;
  std::vector<std::pair<Sub*, int>> rel;  // by stage: segment slot to release
  std::vector<ll> rel_at;                 // stage number that must be consumed, -1: none
  bool fin = false;
  std::vector<Word> words;                // by stage number
  std::vector<std::pair<int, int>> owner; // (subarray, channel) of the step
  // MMA warp.
  ll consumed = 0; bool open = false; std::vector<Group> groups; ll opened = 0;
  // Epilogue.
  ll drained = 0;
};

int main(int argc, char** argv) {
  // grid shape fmt float_chunk rule nsub {N P F T loud slots}
  int a = 1;
  auto next = [&]() { return std::atoi(argv[a++]); };
  int grid = next(); const int shape = next(), fmt = next(), fchunk = next(), rule = next(), nsub = next();
  const bool ints = fchunk == 0;
  std::vector<Sub> subs(nsub);
  for (Sub& s : subs) {
    Geometry g;
    g.N = next(); g.P = next(); g.F = next(); g.T = next();
    g.R = 2 * g.N * g.P; g.Tp = (g.T + 63) / 64 * 64; g.NB = (int64_t)g.N * (g.N + 1) / 2;
    s.loud = next();
    const int slots = next();
    s.g = planar_geometry(g, nullptr);
    s.r = planar_ring(s.g, ints ? 0 : 2, fmt, grid);
    if (slots > 0) s.r.slots = std::min(s.r.slots, std::max(slots, s.r.nseg));
    if (slots < 0) { s.r = planar_ring_whole(s.g, fmt); }
    const int n = s.g.N * s.g.P;
    s.nib = (n + kPlanarBlk - 1) / kPlanarBlk;
    s.nkb = s.g.Tp / 64;
    s.ipc = shape == kPlanar128 ? s.nib * (s.nib + 1) / 2 : pair_items(s.nib);
    s.seg_units = (n + 63) / 64 * s.r.seg_kb;
    s.ready.assign(s.r.slots, 0);
    s.done.assign(s.r.slots, 0);
  }
  const int conv = fmt == XC_PREC_FP8 && ints ? 6 : 4;
  const int stages = fmt == XC_PREC_FP8 && ints ? (shape == kPlanarPair ? 7 : shape == kPlanarWide ? 3 : 5)
                                                : (shape == kPlanar128 ? 3 : 4);
  const int steps = fmt == XC_PREC_HILO ? 3 : fmt != XC_PREC_FP8 && shape == kPlanarWide ? 2 : 1;
  const int sets = fmt == XC_PREC_HILO || shape == kPlanarWide ? 1 : 2;
  std::vector<ll> ib(nsub + 1, 0), ub(nsub + 1, 0);
  for (int i = 0; i < nsub; ++i) {
    ib[i + 1] = ib[i] + (ll)subs[i].g.F * subs[i].ipc;
    ub[i + 1] = ub[i] + (ll)subs[i].g.F * subs[i].r.nseg * subs[i].seg_units;
  }
  ll workers = grid / (shape == kPlanarPair ? 2 : 1);  // CTAs or clusters
  workers = std::min<ll>(workers, ib[nsub]);
  const ll nw = workers * (shape == kPlanarPair ? 2 : 1) * conv;
  int run = ub[nsub] >= 8 * nw ? 2 : 1;
  for (Sub& s : subs) {
    if (s.seg_units % 2) run = 1;
    s.wave = planar_wave((int)workers, s.ipc, s.r.slots, s.g.F);
    if (s.ipc > workers && s.r.slots < s.r.nseg) { std::puts("refused"); return 0; }
  }
  std::vector<Warp> warps(nw);
  for (ll w = 0; w < nw; ++w) { warps[w].u = w * run; warps[w].fin = warps[w].u >= ub[nsub]; }
  std::vector<Cta> ctas(workers);
  for (ll c = 0; c < workers; ++c) {
    ctas[c].it = c;
    ctas[c].rel.resize(stages);
    ctas[c].rel_at.assign(stages, -1);
  }
  auto sub_of = [&](const std::vector<ll>& base, ll v) { int i = 0; while (v >= base[i + 1]) ++i; return i; };
  auto is_ready = [&](Sub& s, int f, int seg) {
    int width; const int G = s.first(f, &width) + seg * width;
    return s.ready[G % s.r.slots] >= (unsigned)(G / s.r.slots + 1) * s.seg_units;
  };
  bool moved = true;
  while (moved) {
    moved = false;
    for (Warp& w : warps) {
      while (!w.fin) {
        const int sb = sub_of(ub, w.u);
        Sub& s = subs[sb];
        const ll v = w.u - ub[sb];
        const int G = (int)(v / s.seg_units), unit = (int)(v % s.seg_units);
        const int full = s.g.F / s.wave, wv = std::min(G / (s.wave * s.r.nseg), full);
        const int width = wv < full ? s.wave : s.g.F - full * s.wave;
        const int seg = (G - wv * s.wave * s.r.nseg) / width, k = unit % s.r.seg_kb;
        const int kb = seg * s.r.seg_kb + k;
        if (kb < s.nkb) {
          const int slot = G % s.r.slots;
          const unsigned gen = G / s.r.slots;
          if (G != w.claimed_G || sb != w.claimed_sb) {
            const bool busy = gen > 0 && s.done[slot] < gen * s.ipc;
            if (busy && w.pend) { w.pend->ready[w.pend_slot] += w.pend_n; w.pend = nullptr; moved = true; }
            if (busy) break;
            w.claimed_G = G; w.claimed_sb = sb;
          }
          if (w.pend && w.pend_run != w.u / run) { w.pend->ready[w.pend_slot] += w.pend_n; w.pend = nullptr; }
          if (!w.pend) { w.pend = &s; w.pend_slot = slot; w.pend_run = w.u / run; w.pend_n = 0; }
          w.pend_n += kb == s.nkb - 1 ? s.r.seg_kb - k : 1;
        }
        w.u += w.u % run != run - 1 ? 1 : 1 + (nw - 1) * run;
        moved = true;
        if (w.u >= ub[nsub]) {
          w.fin = true;
          if (w.pend) w.pend->ready[w.pend_slot] += w.pend_n;
        }
      }
    }
    for (Cta& c : ctas) {
      bool go = true;
      while (go) {
        go = false;
        // Producer: one step, if it can.
        auto release = [&](int s) { ++c.rel[s].first->done[c.rel[s].second]; c.rel_at[s] = -1; go = true; };
        if (!c.fin && c.it >= ib[nsub]) c.fin = true;
        if (c.fin) {
          for (int s = 0; s < stages; ++s) if (c.rel_at[s] >= 0 && c.consumed > c.rel_at[s]) release(s);
        } else {
          const int sb = sub_of(ib, c.it);
          Sub& s = subs[sb];
          const int f = (int)((c.it - ib[sb]) / s.ipc), seg = c.kb / s.r.seg_kb;
          if (c.st == 0 && c.kb % s.r.seg_kb == 0 && !is_ready(s, f, seg)) {
            for (int q = 0; q < stages; ++q) if (c.rel_at[q] >= 0 && c.consumed > c.rel_at[q]) release(q);
          } else if (c.issued < c.consumed + stages) {
            const int q = (int)(c.issued % stages);
            if (c.rel_at[q] >= 0) release(q);
            Word w = {false, false};
            if (c.st == 0) {
              w.start = c.kb == 0;
              if (c.kb == 0) { c.sum = 0; c.f_left = 0; }
              if (ints) {
                const unsigned grow = s.grow(f, seg);
                if (c.kb > 0 && c.sum + grow > (1u << 24)) { w.start = true; c.sum = 0; }
                c.sum += grow;
              } else {
                if (c.f_left == 0) { w.start = true; c.f_left = fchunk; }
                --c.f_left;
                if (fmt == XC_PREC_HILO) w.start = true;
              }
            }
            const bool jlast = c.st + 1 == steps;
            w.end = jlast && (c.kb + 1 == s.nkb || (!ints && (fmt == XC_PREC_HILO || c.f_left == 0)));
            if (jlast && ((c.kb + 1) % s.r.seg_kb == 0 || c.kb + 1 == s.nkb)) {
              int width; const int G = s.first(f, &width) + seg * width;
              c.rel[q] = {&s, G % s.r.slots};
              c.rel_at[q] = c.issued;
            }
            c.words.push_back(w);
            c.owner.push_back({sb, f});
            ++c.issued;
            go = true;
            if (++c.st == steps) { c.st = 0; if (++c.kb == s.nkb) { c.kb = 0; c.it += workers; } }
          }
        }
        // MMA warp: one step.
        if (c.consumed < c.issued) {
          const Word w = c.words[c.consumed];
          const std::pair<int, int> o = c.owner[c.consumed];
          if (w.start && c.open) { c.groups.push_back({o.first, o.second}); c.open = false; go = true; }
          if (w.start && c.opened - c.drained >= sets) {
            // waits for a drain
          } else {
            if (w.start) { c.open = true; ++c.opened; }
            ++c.consumed;
            go = true;
            if (w.end) { c.groups.push_back({o.first, o.second}); c.open = false; }
          }
        }
        // Epilogue: one group.  The rule under test: does it first wait for the
        // whole channel?
        if (c.drained < (ll)c.groups.size()) {
          const Group g = c.groups[c.drained];
          Sub& s = subs[g.sb];
          bool ok = true;
          if (rule == 1)
            for (int seg = 0; seg < s.r.nseg; ++seg) ok = ok && is_ready(s, g.f, seg);
          if (ok) { ++c.drained; go = true; }
        }
        moved = moved || go;
      }
    }
  }
  bool all = true;
  for (Warp& w : warps) all = all && w.fin;
  for (Cta& c : ctas) all = all && c.fin && c.consumed == c.issued && c.drained == (ll)c.groups.size();
  std::puts(all ? "done" : "stuck");
  return 0;
}
"""
FP16, HILO, FP8 = 0, 1, 2
S128, PAIR, WIDE = 0, 1, 2


@pytest.fixture(scope="module")
def model(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not available")
    d = tmp_path_factory.mktemp("ring")
    src = d / "ring.cpp"
    src.write_text(HARNESS)
    exe = d / "ring"
    subprocess.run([gxx, "-std=c++17", "-O2", "-I", CSRC, "-I", os.path.join(ROOT, "include"), str(src), "-o",
                    str(exe)], check=True)

    def run(subs, shape=S128, fmt=FP16, fchunk=0, whole_channel=False, grid=152):
        args = [grid, shape, fmt, fchunk, int(whole_channel), len(subs)] + [v for s in subs for v in s]
        return subprocess.run([str(exe)] + [str(v) for v in args], check=True, capture_output=True,
                              text=True).stdout.strip()
    return run


# (N, P, F, T, max |x|, shape): channels whose ring share is less than what two
# exact chunks (one on 128 x 256 items) leave unread.
STALLS = [(72, 2, 64, 3584, 128, S128), (100, 2, 64, 9216, 50, S128), (160, 2, 64, 4096, 128, S128),
          (256, 2, 64, 4608, 128, S128), (256, 2, 64, 10240, 50, PAIR), (300, 2, 64, 7168, 80, S128),
          (512, 2, 64, 5632, 80, WIDE), (128, 2, 256, 4096, 128, S128), (256, 2, 64, 8192, -128, S128)]


@pytest.mark.parametrize("size", STALLS, ids=lambda s: "N%d_P%d_F%d_T%d_m%d_shape%d" % s)
def test_epilogue_waits_for_accumulators_only(size, model):
    sub, shape = size[:5] + (0,), size[5]
    assert model([sub], shape, whole_channel=True) == "stuck"
    assert model([sub], shape) == "done"


def test_random_sizes_never_stall(model):
    """Every shape, operand format and loudness, rings cut down to one channel,
    batches; 152 SMs and fewer."""
    rng = random.Random(11)
    for i in range(60):
        shape = rng.choice([S128, S128, PAIR, WIDE])
        ints = rng.random() < 0.75
        fmt = rng.choice([FP16, FP16, FP8] if ints else ([FP16, HILO] if shape != WIDE else [FP16]))
        subs = []
        for _ in range(rng.choice([1, 1, 3]) if ints and fmt == FP16 else 1):
            N, P = rng.choice([3, 40, 65, 100, 160, 256, 449, 700]), rng.choice([1, 2])
            nib = (N * P + 127) // 128
            T = rng.choice([1, 64, 513, 2112, 4608, 9216, 20000])
            F = rng.randint(1, max(1, min(90, 400000 // (nib * nib * (T // 64 + 1)))))
            subs.append((N, P, F, T, rng.choice([0, 20, 128, -128, 1000 + i]), rng.choice([0, 0, 1, -1])))
        grid = rng.choice([152, 152, 148, 20, 2])
        got = model(subs, shape, fmt, 0 if ints else rng.choice([1, 8, 16, 4096]), grid=grid)
        assert got == "done", (subs, shape, fmt, grid, got)
