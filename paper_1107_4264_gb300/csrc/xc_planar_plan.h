// xc_planar_plan.h -- sizes of the planar tensor-core X-engine that the host
// decides: channel packing, tile shape, operand ring and waves (plain C++).
#pragma once

#include <algorithm>
#include <cstdint>

#include "xc.h"
#include "xc_internal.h"

namespace xc {

// Tile shapes: 128 x 128 blocks on single CTAs, two blocks sharing a column
// block on a CTA pair (tcgen05 cta_group::2), two blocks sharing a row block on
// one CTA (N = 256 MMAs).
// 128 x 128 is the one a call takes unless it asks for another.  128 x 256
// items are faster for large arrays with long, quiet 8-bit integrations (512
// stations x 2 pols, F=64, T=4096: 0.69 against 0.77 ms), but their
// accumulators fill TMEM, so the MMAs stop for every drain of an exact chunk:
// at |x| up to 80 there 2.89 against 0.93 ms, at full scale 5.16 against 1.14;
// and how loud the samples are is not known at the launch.
enum : int { kPlanar128 = 0, kPlanarPair = 1, kPlanarWide = 2 };
constexpr int kPlanarBlk = 128;  // inputs per block
// Samples per K-block and converter unit (8-bit input arrives by TMA in
// 128-row x 1 x kPlanarUnitT boxes).
constexpr int kPlanarUnitT = 64;
constexpr int kMaxRingSlots = 1024;

// Small arrays (n = N P <= 64 inputs): k consecutive channels, k the largest
// divisor of F with k n <= 128, are correlated as one virtual channel of k N
// stations.  The input [T][F][n] is the same memory as [T][F / k][k n], so
// nothing moves; one 128 x 128 block then holds the k channels' own blocks on
// its diagonal.  Returns that virtual geometry and k (1 for larger arrays).
inline Geometry planar_geometry(const Geometry& g, int* pack) {
  int k = 1;
  const int64_t n = static_cast<int64_t>(g.N) * g.P;
  if (n <= kPlanarBlk / 2) {
    for (int c = static_cast<int>(kPlanarBlk / n); c >= 2; --c) {
      if (g.F % c == 0) {
        k = c;
        break;
      }
    }
  }
  Geometry v = g;
  v.N = g.N * k;
  v.F = g.F / k;
  v.R = g.R * k;
  v.NB = static_cast<int64_t>(v.N) * (v.N + 1) / 2;
  if (pack) *pack = k;
  return v;
}

// The planar engine's operand ring: a channel's K-blocks are split into nseg
// segments of seg_kb (the last one shorter), and a slot holds one segment's
// operand tiles.  Formats are XC_PREC_* (8-bit input: in_dtype 0).
struct PlanarRing {
  int seg_kb, nseg, slots;
  int64_t slot_bytes;
};
inline PlanarRing planar_ring_of(const Geometry& g, int fmt, int seg_kb) {
  const int64_t nib = (static_cast<int64_t>(g.N) * g.P + kPlanarBlk - 1) / kPlanarBlk;
  const int per_sample = fmt == XC_PREC_HILO ? 4 : fmt == XC_PREC_FP8 ? 1 : 2;  // bytes of one plane
  PlanarRing r;
  r.seg_kb = seg_kb;
  r.nseg = (g.Tp / kPlanarUnitT + seg_kb - 1) / seg_kb;
  r.slots = 1;
  r.slot_bytes = 2 * per_sample * static_cast<int64_t>(seg_kb) * nib * (kPlanarBlk * kPlanarUnitT);
  return r;
}

// One segment per channel (the least memory that works: one slot).
inline PlanarRing planar_ring_whole(const Geometry& g, int fmt) {
  return planar_ring_of(g, fmt, g.Tp / kPlanarUnitT);
}

// Segments of at most 8 K-blocks (512 samples; half as many with hi/lo
// operands, which take twice the bytes) and 60 MiB of ring, so that it stays
// in the 129 MB L2 beside the streams.  Measured (8-bit input, ms):
//   K-blocks per segment       16     8     4
//     N=100 F=512  T=1000   0.243 0.207 0.203
//     N=256 F=1024 T=1000   0.987 0.969 0.988
//     N=200 F=256  T=512    0.144 0.144 0.150
//   ring                   50 MiB 60 MiB 75 MiB 90 MiB 120 MiB 250 MiB
//     N=256 F=1024 T=1000   1.028  0.977  1.044  1.100   1.144
//     N=256 F=256  T=4096          1.104         1.004   1.061   1.099
//     N=256 F=64   T=8192          0.671         0.604   0.605   0.602
//     N=512 F=64   T=4096          0.809         0.822   0.830   0.824
// So 90 MiB when the channels of a wave take more than 80 MiB (8-bit input:
// the float converters are too slow to fill it).
inline PlanarRing planar_ring(const Geometry& g, int in_dtype, int fmt, int grid) {
  const int seg = fmt == XC_PREC_HILO ? 4 : 8;
  const int nkb = g.Tp / kPlanarUnitT;
  const int parts = (nkb + seg - 1) / seg;
  PlanarRing r = planar_ring_of(g, fmt, (nkb + parts - 1) / parts);
  const int64_t nib = (static_cast<int64_t>(g.N) * g.P + kPlanarBlk - 1) / kPlanarBlk;
  const int64_t wave = std::max<int64_t>(1, grid / (nib * (nib + 1) / 2));
  int64_t mib = 60;
  if (in_dtype == 0 && wave * r.nseg * r.slot_bytes > (80ll << 20)) mib = 90;
  int64_t n = std::min<int64_t>((mib << 20) / r.slot_bytes, kMaxRingSlots);
  n = std::max<int64_t>(n, std::max<int64_t>(4, r.nseg + 4));
  r.slots = static_cast<int>(std::min<int64_t>(n, static_cast<int64_t>(g.F) * r.nseg));
  return r;
}

// Ring slots that the counters of a handle have to serve: the most that any
// operand format of its input type asks for.  (A ring is at least nseg + 4
// slots, whatever kMaxRingSlots says, and hi/lo segments are half as long.)
inline int planar_max_slots(const Geometry& g, int in_dtype, int grid) {
  int n = planar_ring(g, in_dtype, XC_PREC_FP16, grid).slots;
  n = std::max(n, planar_ring(g, in_dtype, XC_PREC_FP8, grid).slots);
  if (in_dtype != 0) n = std::max(n, planar_ring(g, in_dtype, XC_PREC_HILO, grid).slots);
  return n;
}

// Channels per wave: as many as there are CTAs (clusters: `workers`) for their
// items, and no more than half the ring's slots.  (N=256 F=64 T=8192 on a 60 MiB
// ring: 0.686 ms, and 1.150 ms with one channel to a wave.)
inline int planar_wave(int workers, int items_per_channel, int ring_slots, int F) {
  return std::max(1, std::min({workers / items_per_channel, ring_slots / 2, F}));
}

}  // namespace xc
