#pragma once
// xc_planar_kernel.cuh -- fused persistent tensor-core X-engine, planar
// complex form: the kernel template, shared by the translation units that
// instantiate its single-CTA (xc_planar.cu) and CTA-pair (xc_planar_pair.cu)
// variants.
//
// Eq. (outer) of Sec. 2.1 per channel f: V_f = sum_t x_f(t) x_f(t)^H over
// n = N*P complex inputs.  With the real and imaginary parts of the inputs
// as separate fp16 operand planes Xr, Xi (n rows x T samples, K-major),
//
//     Re V = Xr Xr^T + Xi Xi^T,      Im V = Xi Xr^T - Xr Xi^T,
//
// so a 128 x 128 block of V (rows a, columns b) is four tcgen05 MMAs per
// 16-sample step into two TMEM accumulators,
//     D_re += Ar Br^T,  D_re += Ai Bi^T,  D_im += Ai Br^T,  D_im += Ar (-Bi)^T,
// the last with the instruction descriptor's negate-B bit.  Four operand
// tiles feed 4 MMAs (half the shared-memory and L2 bytes per MAC of the
// interleaved real form) and every TMEM column is a finished visibility
// component: the epilogue converts and stores, with no lane exchange.
//
// Exact 8-bit input: int8 is exact in fp16, products are exact in fp32, and
// every partial sum of an accumulator is an integer bounded by the sum of
// |products| so far: at most 2 m^2 per sample, m = max |x| of the channel.
// The converters record m per channel; a chunk of S samples with
// 2 m^2 S <= 2^24 is exact in fp32 in any summation order (S >= 512 for any
// int8 data, the whole integration for typical 4-6 bit signal levels).  Each
// chunk is drained into int32 and added into the output (stored for the
// first chunk).  Float input accumulates in fp32 over the whole integration.
//
// Float input (Sec. 5 leaves its precision open): each (channel, input) gets
// a power-of-two scale 2^e from a pre-pass over the integration (max
// component of g x), so y 2^-e spans the operand format's range and the
// epilogue multiplies by 2^(e_a + e_b) exactly.  Three operand formats:
//   FP16   one fp16 plane pair, 4 MMAs per 16 samples;
//   HI/LO  y 2^-e = h + l with h = fp16(.) and l = fp16(. - h); the ring
//          holds H and L tiles and each 64-sample block runs three steps
//          (H H^T, L H^T, H L^T; the l l^T term is dropped), 3x the MMAs;
//   FP8    e4m3 planes (kind::f8f6f4, K = 32), half the operand bytes.
// Optionally (FP64 block sums) the fp32 accumulator is drained every
// T_blk samples into a float64 running sum; the output is its rounding.
//
// Blocks (Sec. 4.2): 128 x 128 blocks of V on or below the block diagonal,
// g = by(by+1)/2 + bx; block edges fall on station boundaries (128 inputs =
// 128/P stations).  Diagonal blocks load one pair of planes for both
// operands and store only their lower station triangle (Sec. 4.4).
//
// Operand formation (Sec. 4.1 input order, Sec. 5 8-bit samples): converter
// warps form each channel's planes once into a ring in global memory that
// stays in L2; the blocks of a channel read it back with bulk copies.  The
// ring's unit is a segment of a channel (seg_kb K-blocks of 64 samples, all
// its inputs); the channels at work at one time (a wave) are brought a segment
// each in turn, so the ring's size follows neither the channels' length nor
// how many of them are in flight (seg_first).
// The ring holds operand tiles exactly as the MMA reads them: per (slot,
// K-block, 128-input block) the two planes' tiles of 128 inputs x four 16-byte
// K chunks (8 KiB) in the no-swizzle K-major canonical layout, K inside:
// [8-input group][chunk][8 inputs][16 B], so a stage is one contiguous copy
// per operand, inputs 0..63 and 64..127 of a tile are its two contiguous
// halves, and the 8 x 16 B core matrix that four converter lanes write is one
// whole line.  8-bit input arrives by TMA in 128-row x 64-sample boxes (other
// types likewise; rows that TMA cannot stride by plain loads, 8-bit ones as
// 32-bit words); each converter warp works through its own stream of units.  Ring protocol:
//   ready[slot] counts converted units (64 inputs x 64 samples); segment G
//     (generation G / slots of slot G % slots) is complete at
//     ready >= (gen + 1) * units_per_segment;
//   done[slot] counts work items whose MMAs have read the segment; slot s may
//     take segment G once done >= gen(G) * items_per_channel.
// A segment waits for segments of lower number only, and a work item for
// segments of its own channel, one after the other: the producer for each when
// it comes to it, the MMA warp for stages and drained accumulators, and the
// epilogue for full accumulators alone (stage_acc, acc_last), never for a
// segment, so a drain needs nothing that the MMAs before it did not.  All CTAs
// are co-resident and each has at most one item of a wave, so the items of the
// lowest number not yet read are at work or come next once the waves before are
// done: the ring cannot deadlock, however little of a wave it holds.  (When a
// channel has more items than there are CTAs, a wave is one channel and the
// ring holds all its segments.)  Every wait is bounded regardless.
//
// CTA roles (persistent, one CTA per SM, channel-major items):
//   warp 0      producer: 3 stages x (Ar, Ai, Br, Bi) of 64 samples (bulk copies);
//               releases segments
//   warp 1      MMA issuer; owns TMEM (2 sets x {D_re, D_im} x 128 columns)
//   warps 2..5  epilogue
//   warps 6..9  converters
// What bounds it: the converters' and the epilogue's stores share the SM's
// shared-memory path with the MMAs' operand reads.  Alone, the stage copies and
// MMAs of a 64-sample step take 1114 cycles (1024 is the tensor rate); with 4
// warps storing 64 KiB of tiles per 6500 cycles some 200 more, and 300 more
// again with the epilogue's stores as well.  From a ring of whole channels, one
// thread per CTA that walked the items and issued, a wait of the epilogue for
// the channel's maximum and an FP64 square root and several divisions per item
// and role to now: 1.07 -> 0.99-1.01 ms on the 256-station array (1024 channels
// of 1000 samples), 0.196 -> 0.139 ms for 200 stations, 256 channels of 512, and
// 1.02 -> 0.54 ms at 2048 channels of 125 samples.
//
// CTA pairs (PAIR = true, tcgen05 cta_group::2, clusters of two CTAs): one
// item is two 128 x 128 blocks sharing their column block b, computed by one
// 256 x 128 MMA per step over the pair.  CTA k stages the 128 rows of its
// own row block a_k (Ar, Ai tiles) and inputs 64k .. 64k + 63 of block b (the
// k-th halves of the Br, Bi tiles); the leader (rank 0) issues the MMAs, each
// SM's TMEM receives its row block's D_re, D_im.  Per SM the shared-memory
// operand reads per MAC drop by a quarter (A plus half of B per 128 x 128
// product instead of A plus B) and B is staged once for two blocks.
// Pairing (pair_coords): in column block c the blocks of rows c, c+1, ...
// pair off from the diagonal down; the odd one out of a column, (nib-1, c),
// is taken transposed, as rows c times columns nib-1 (its mirror, V[c][nib-1]
// = conj(V[nib-1][c])^T), so the leftovers of all columns share column block
// nib-1 and pair among themselves: ceil(blocks / 2) items per channel, at
// most one CTA of one item idle.  A transposed block is stored as its mirror.
// Hand-offs between the two CTAs:
//   full[s]   local completion of stage s's copies (each CTA)
//   pfull[s]  leader: the peer's relay thread forwards its full[s]
//   empty[s]  both: the leader's commit, multicast, once the MMAs reading
//             stage s in both SMs have completed
//   accf[b]   both: accumulator b holds a finished group (multicast commit)
//   acce[b]   leader: 8 epilogue warps (4 per CTA) have read accumulator b
#include <cuda.h>
#include <cuda_fp16.h>
#include <cuda_fp8.h>

#include <algorithm>
#include <cstring>
#include <type_traits>

#include "xc_launch.h"
#include "xc_ptx.cuh"

namespace xc {
namespace {

constexpr int kBlk = 128;      // complex inputs per block side
constexpr int kBK = 64;        // samples per stage
constexpr int kNumEpiWarps = 4;
constexpr int kNumConvWarps = 4;
constexpr int kThreads = 32 * (2 + kNumEpiWarps + kNumConvWarps);
constexpr uint32_t kTmemCols = 512;         // 2 sets x (D_re, D_im) x 128
constexpr int kUnitRows = 128;  // converter unit: 128 real rows (64 inputs) x kUnitT samples
constexpr int kUnitT = kPlanarUnitT;
static_assert(kUnitT == kBK, "a unit covers one 64-sample K-block");
constexpr uint32_t kCoreBytes = 8 * 16;  // one core matrix: 8 inputs x 16 bytes
constexpr int kConvBufBytes = kUnitRows * kUnitT;  // int8 staging per converter warp

// Tile shapes (XC_TILE_*): 128 x 128 blocks on single CTAs; two blocks
// sharing a column block on a CTA pair (256 x 128 MMAs, cta_group::2); two
// blocks sharing a row block on one CTA (128 x 256 MMAs).
enum : int { kShape128 = 0, kShapePair = 1, kShapeWide = 2 };

enum : int { kFmtF16 = 0, kFmtHiLo = 1, kFmtF8 = 2 };

// The stage plan of 8-bit input on e4m3 operands, whose conversion costs the
// most per byte while its MMAs take half the time: half-size stages, and six
// converter warps instead of four (float input keeps the fp16 plan: its
// converters gain nothing from more warps and spill more registers).
template <int FMT, int DT>
constexpr bool f8_int8_plan() {
  return FMT == kFmtF8 && DT == 0;
}
template <int FMT, int DT>
constexpr int conv_warps() {
  return f8_int8_plan<FMT, DT>() ? 6 : kNumConvWarps;
}
template <int FMT, int DT>
constexpr int threads_of() {
  return 32 * (2 + kNumEpiWarps + conv_warps<FMT, DT>());
}

// Operand formats.  A tile holds kChunks 16-byte K chunks of 128 inputs: the
// 64 samples of a K-block, or half of them for fp16 operands on 128 x 256
// items, whose two 96 KiB stages would leave little to run ahead with (a
// stage is one tile per plane; on the other shapes finer stages lose more to
// a stage's fixed cost in the MMA warp than they give: 128 x 128 on the
// 256-station array 1.03 against 0.98 ms).
template <int FMT, int SHAPE>
struct FmtT {
  static constexpr int kChunks = FMT == kFmtF8 || SHAPE == kShapeWide ? 4 : 8;
  static constexpr int kTile = kBlk * 16 * kChunks;
  static constexpr int kSplit = (FMT == kFmtF8 ? 4 : 8) / kChunks;  // tiles per plane and K-block
  static constexpr int kHalves = FMT == kFmtHiLo ? 3 : 1;  // operand pairs per K-block (H H, L H, H L)
  static constexpr int kSteps = kHalves * kSplit;          // stages per K-block
  // A K-block of one input block in the ring: [kSplit][plane] tiles.
  static constexpr int kKbBytes = kSplit * 2 * kTile;
  // Bytes between 8-input groups of a tile (the descriptor's stride offset);
  // core matrices adjacent in K are kCoreBytes apart (its leading offset).
  static constexpr uint32_t kSbo = kChunks * kCoreBytes;
};

// Shared-memory plan per shape and operand format: stages of (Ar, Ai, Br,
// Bi) tiles; (Ar, Ai, half Br, half Bi) on pairs; (Ar, Ai, Br Br', Bi Bi')
// for 128 x 256; then the converters' staging buffers and the barriers.
// e4m3 tiles are half the size of fp16 ones: for 8-bit input, more stages
// and two more converter warps fit in the same bytes.
template <int SHAPE, int FMT, int DT>
struct Cfg {
  static constexpr bool kF8 = f8_int8_plan<FMT, DT>();
  static constexpr int kStages = kF8 ? (SHAPE == kShapePair ? 7 : (SHAPE == kShapeWide ? 3 : 5))
                                     : (SHAPE == kShapePair ? 4 : (SHAPE == kShapeWide ? 4 : 3));
  static constexpr int kStageBytes =
      (SHAPE == kShapePair ? 3 : (SHAPE == kShapeWide ? 6 : 4)) * FmtT<FMT, SHAPE>::kTile;
  static constexpr int kConvOff = kStages * kStageBytes;
  static constexpr int kBarOff = kConvOff + conv_warps<FMT, DT>() * kConvBufBytes;
  // full, empty (and pfull) per stage; accf, acce x 2; drain; one per converter
  static constexpr int kNumBars = (SHAPE == kShapePair ? 3 : 2) * kStages + 5 + conv_warps<FMT, DT>();
  // then the TMEM address, the abort flag, one word per stage (stage_acc) and
  // one per accumulator set (acc_last)
  static constexpr int kSmemBytes = kBarOff + kNumBars * 8 + 8 + 4 * (kStages + 2) + 1024;
  static_assert(kSmemBytes <= 232448, "shared memory budget");
};

// Byte offset of (input row, 16-byte K chunk of the K-block) from the K-block's
// first tile of a plane.
template <int FMT, int SHAPE>
__device__ __forceinline__ uint32_t tile_off(int row, int chunk) {
  return static_cast<uint32_t>(chunk / FmtT<FMT, SHAPE>::kChunks) * (2 * FmtT<FMT, SHAPE>::kTile) +
         static_cast<uint32_t>(row >> 3) * FmtT<FMT, SHAPE>::kSbo +
         static_cast<uint32_t>(chunk % FmtT<FMT, SHAPE>::kChunks) * kCoreBytes + static_cast<uint32_t>(row & 7) * 16u;
}

struct Params {
  Geometry g;
  int n;               // complex inputs per channel = N * P
  const void* in;
  void* out;
  int accumulate;
  int ntiles;          // lower blocks per channel
  int ipc;             // work items per channel: ntiles, or pair items (CTA pairs)
  long long nitems;    // ipc * F
  int nkb;             // Tp / 64
  int is_int;          // 8-bit input: exact chunks from the channel's max |x|
  unsigned* amax;      // [F][nseg] max |x| per channel segment (8-bit input), zeroed by the host
  const float2* gains; // [n] complex gains applied to float input (y = g x), or NULL
  const unsigned* in_amax;  // [F][n] max component of g x (float bits), float input
  double* acc64;       // FP64 block sums: running visibility sums (output layout), or NULL
  int f_chunk_kb;      // float input: K-blocks per fp32 accumulation chunk
  uint8_t* ring;       // tiles [slots][nkt][nib][split][2][chunks][128][16 B]
  int nkt;             // K-tiles per plane per input block of a slot (seg_kb or 2 seg_kb)
  int nib;             // 128-input blocks per channel
  int seg_kb, nseg;    // K-blocks per ring segment; segments per channel
  int ring_slots;      // segment slots, at least nseg
  unsigned* ready;     // [ring_slots]
  unsigned* done;      // [ring_slots]
  // Converter units per segment: seg_kb for each 64-input half block that holds
  // an input.  The last block's upper half is never written when it holds none:
  // whatever the ring holds there only reaches rows and columns of the
  // accumulators past n, which no one reads.  (A 48-input array converts half
  // as many units, 400 inputs seven eighths.)
  int seg_units;
  // Channels go through the ring in waves of `wave` (the last one of
  // wave_last, from segment number last_base on): see seg_first.
  int wave, wave_segs, wave_full, wave_last, last_base;
  unsigned mag_kb, mag_wave, mag_wsegs, mag_last, mag_slots;  // fast_div magics
  int run;  // units per run (the same in all subarrays)
  // From one of a converter warp's runs to its next (run * converter warps
  // units on): step_seg segments and step_rem units, and step_seg as
  // ring generations and slots.
  int step_seg, step_rem, step_gen, step_slot;
  // From one of a CTA's (cluster's) items to its next: channels and items.
  int it_step_f, it_step_i;
  int tma_in;          // input staged by TMA (rows are a multiple of 16 bytes)
  unsigned long long timeout_ns;
  int* status;
  int test_no_publish;  // test hook: converted units are never published
  // Small arrays: `pack` consecutive channels form one virtual channel of
  // pack * Nr stations (g, n, F above are the virtual geometry; the input
  // [T][F][n] is the same memory as [T][F / pack][pack * n]).  The epilogue
  // keeps only each real channel's own block and stores it at real indices.
  int pack;
  int Nr;              // real stations per channel
  int64_t NBr;         // real baselines per channel
  int gain_n;          // real inputs per channel (gains are indexed a mod gain_n)
};

// One launch over up to kMaxSub subarrays (Sec. 4.2's channel-major raster
// extended across subarrays): items and converter units are numbered
// subarray by subarray; item_base / unit_base are their prefix sums.  Each
// subarray has its own ring region and counters.
struct Batch {
  CUtensorMap maps[kMaxSub];  // 8-bit input of each subarray (read when tma_in)
  Params sub[kMaxSub];
  long long item_base[kMaxSub + 1];
  long long unit_base[kMaxSub + 1];
  int nsub;
};
static_assert(sizeof(Batch) <= kBatchArgBytes && alignof(Batch) <= 128, "batch parameter block");

// Subarray holding global index i, starting the search at cursor s (every
// role walks its items and units in increasing order).  Single-subarray
// launches (MULTI = false) index subarray 0 at compile time.
// End of a prefix-sum table (compile-time index for single launches).
template <bool MULTI>
__device__ __forceinline__ long long table_end(const long long* base, int nsub) {
  if constexpr (!MULTI) {
    return base[1];
  } else {
    return base[nsub];
  }
}

template <bool MULTI>
__device__ __forceinline__ int advance_sub(const long long* base, int nsub, long long i, int s) {
  if constexpr (!MULTI) {
    return 0;
  } else {
    while (s + 1 < nsub && i >= base[s + 1]) ++s;
    return s;
  }
}

// ------------------------------------------------------------ global sync

__device__ __forceinline__ unsigned ld_acquire(const unsigned* p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void red_release_add(unsigned* p, unsigned v) {
  asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
__device__ __forceinline__ void fence_proxy_async_global() {
  asm volatile("fence.proxy.async.global;" ::: "memory");
}

__device__ __noinline__ bool wait_counter(const unsigned* p, unsigned target, const Params& prm,
                                          volatile int* abort_flag) {
  if (ld_acquire(p) >= target) return true;
  const uint64_t t0 = ptx::globaltimer();
  for (uint32_t it = 1;; ++it) {
    __nanosleep(64);
    if (ld_acquire(p) >= target) return true;
    if ((it & 15u) == 0) {
      if (*abort_flag) return false;
      if (*reinterpret_cast<volatile int*>(prm.status) != 0) {
        *abort_flag = 1;
        return false;
      }
      if (ptx::globaltimer() - t0 > prm.timeout_ns) {
        *abort_flag = 1;
        atomicOr(prm.status, kStatusTimeout);
        return false;
      }
    }
  }
}

// Is a wait that began at t0 over (another role gave up, or the time is up)?
// For loops that do something else in between.
__device__ __noinline__ bool wait_given_up(const Params& prm, uint64_t t0, volatile int* abort_flag) {
  if (*abort_flag) return true;
  const bool late = ptx::globaltimer() - t0 > prm.timeout_ns;
  if (!late && *reinterpret_cast<volatile int*>(prm.status) == 0) return false;
  *abort_flag = 1;
  if (late) atomicOr(prm.status, kStatusTimeout);
  return true;
}

// A work item: its number in the launch, its subarray, channel and number in
// the channel.  Stepped from item to item without divisions (and the block
// coordinates below come from a float square root: the FP64 one of
// tri_coords cost every role some thousand cycles per item).
struct Item {
  long long it;
  int sb, f, i;
};
template <bool MULTI>
__device__ __forceinline__ void item_locate(const Batch& bt, Item& x) {
  x.sb = advance_sub<MULTI>(bt.item_base, bt.nsub, x.it, x.sb);
  const Params& p = bt.sub[x.sb];
  const long long v = x.it - bt.item_base[x.sb];
  x.f = static_cast<int>(v / p.ipc);
  x.i = static_cast<int>(v - static_cast<long long>(x.f) * p.ipc);
}
template <bool MULTI>
__device__ __forceinline__ Item item_start(const Batch& bt, long long it, long long nitems) {
  Item x = {it, 0, 0, 0};
  if (it < nitems) item_locate<MULTI>(bt, x);
  return x;
}
template <bool MULTI>
__device__ __forceinline__ void item_step(const Batch& bt, Item& x, long long step, long long nitems) {
  x.it += step;
  if (x.it >= nitems) return;
  if (MULTI && x.it >= bt.item_base[x.sb + 1]) {
    item_locate<MULTI>(bt, x);
    return;
  }
  const Params& p = bt.sub[x.sb];
  x.f += p.it_step_f;
  x.i += p.it_step_i;
  if (x.i >= p.ipc) {
    x.i -= p.ipc;
    ++x.f;
  }
}

// Lower block i of a channel: row by, column bx (Sec. 4.2's inverse map, the
// float estimate corrected with exact integers).
__device__ __forceinline__ void block_coords(int i, int* bx, int* by) {
  long long y = static_cast<long long>((__fsqrt_rn(8.f * static_cast<float>(i) + 1.f) - 1.f) * 0.5f);
  while (y * (y + 1) / 2 > i) --y;
  while ((y + 1) * (y + 2) / 2 <= i) ++y;
  *by = static_cast<int>(y);
  *bx = static_cast<int>(i - y * (y + 1) / 2);
}

// This CTA's share of work item `it` (local to its subarray): channel f,
// row block a and column block b (128 x 256 items: column blocks b and b2,
// b2 = -1 when the item holds one block); idle: the second CTA of a
// one-block pair item.  A block with a column block above its row block
// (b > a) is computed as is and stored as its mirror.
struct Blk {
  int f, a, b, b2;
  bool idle;
};
template <int SHAPE>
__device__ __forceinline__ Blk item_block(const Params& p, const Item& x, uint32_t rank) {
  Blk k;
  k.f = x.f;
  k.b2 = -1;
  k.idle = false;
  if constexpr (SHAPE == kShape128) {
    block_coords(x.i, &k.b, &k.a);
    (void)p;
    (void)rank;
  } else {
    int a0, a1, b, single;
    pair_coords(x.i, p.nib, &a0, &a1, &b, &single);
    if constexpr (SHAPE == kShapePair) {
      k.a = rank ? a1 : a0;
      k.b = b;
      k.idle = rank && single;
    } else {
      // The pair schedule transposed: the common block is the row block;
      // the column blocks ascend, so a ragged last block comes second.
      (void)rank;
      k.a = b;
      k.b = single ? a0 : min(a0, a1);
      k.b2 = single ? -1 : max(a0, a1);
    }
  }
  return k;
}

// x / d for a run-time d, with mag = floor(2^32 / d) (2^32 - 1 for d = 1):
// the product's high word is the quotient or one less.
__device__ __forceinline__ int fast_div(int x, int d, unsigned mag) {
  const int q = static_cast<int>(__umulhi(static_cast<unsigned>(x), mag));
  return x - q * d >= d ? q + 1 : q;
}

// Segments are numbered (and take ring slots, in turn) wave by wave, within a
// wave segment by segment, within a segment channel by channel: the channels
// that are worked on at the same time arrive together, a segment each, so the
// ring need not hold whole channels of a long integration.  Channel f's
// segments are numbers first, first + *width, first + 2 *width, ...
// A wave holds no more work items than there are CTAs (or is one channel), so
// all its items are at work at the same time and none waits for a segment
// whose slot is held for an item that has yet to start.
__device__ __forceinline__ int seg_first(const Params& p, int f, int* width) {
  const int w = fast_div(f, p.wave, p.mag_wave);
  *width = w < p.wave_full ? p.wave : p.wave_last;
  return w * p.wave_segs + f - w * p.wave;
}

// 8-bit input: how much a partial sum can grow over one K-block of segment G
// (its number in the subarray), from the segment's max |x|; at most 2^21.
// Called after the segment is known to be converted.  A chunk is exact in
// fp32 while its K-blocks' growths sum to at most kExactSum.
constexpr unsigned kExactSum = 1u << 24;
__device__ __forceinline__ unsigned kblock_growth(const Params& p, int G) {
  const unsigned m = *reinterpret_cast<volatile const unsigned*>(p.amax + G);
  return 2u * m * m * kBK;
}

// -------------------------------------------------------------- converter

// How a kernel's converters read their input: 8-bit in TMA boxes, 8-bit in words
// (rows that TMA cannot stride), or float (either way).  One 8-bit form per
// kernel: with both in one, the words' 64 registers spill in the kernel whose
// input is aligned too (288 bytes of stores, none without them).
enum : int { kInTma = 0, kInWords = 1, kInFloat = 2 };

// fp16x2 of (component j of sample a, component j of sample b), 8-bit input.
__device__ __forceinline__ uint32_t pair_i8(uint32_t a, uint32_t b, uint32_t j) {
  // Byte j of a into byte 0 and byte j of b into byte 2; 0x6400 | (x ^ 0x80)
  // is the fp16 value 1152 + x, so subtracting 1152 gives x exactly.
  uint32_t d = __byte_perm(a, b, j | ((j + 4u) << 8));
  d = (d & 0x00FF00FFu) ^ 0x64806480u;
  __half2 h = *reinterpret_cast<__half2*>(&d);
  h = __hsub2(h, __half2(__float2half_rn(1152.f), __float2half_rn(1152.f)));
  return *reinterpret_cast<uint32_t*>(&h);
}

// Byte address of the first tile of (slot, plane, K-tile kt, ib) in the ring: a
// K-tile is a K-block's tiles, [kSplit][plane], so that the two planes of a
// stage lie side by side (one copy brings both).
template <int FMT, int SHAPE>
__device__ __forceinline__ uint8_t* ring_tile(const Params& p, int slot, int plane, int kt, int ib) {
  return p.ring + ((static_cast<int64_t>(slot) * p.nkt + kt) * p.nib + ib) * FmtT<FMT, SHAPE>::kKbBytes +
         plane * FmtT<FMT, SHAPE>::kTile;
}

// Power-of-two scale exponent e for an input whose largest component is
// `bits` (fp32 bits): max |y| 2^-e lies in [2^14, 2^15) for the fp16 forms
// and in (2^7, 448] for e4m3.  Zero or subnormal maxima are not scaled;
// e is clamped to [-60, 60] so that 2^(e_a + e_b) is a normal float.
template <int FMT>
__device__ __forceinline__ int scale_exp(unsigned bits) {
  const int E = static_cast<int>((bits >> 23) & 0xffu);
  if (E == 0) return 0;
  int e = E - 127 - (FMT == kFmtF8 ? 8 : 14);
  if (FMT == kFmtF8 && (bits & 0x7fffffu) > 0x600000u) ++e;  // 256 (1 + m) > 448
  return max(-60, min(60, e));
}
__device__ __forceinline__ float exp2i(int e) { return __int_as_float((127 + e) << 23); }

// A converter unit: 64 inputs (half block hb) x one K-block (k of its
// segment) of segment number G.  Units are numbered segment by
// segment, half block by half block, K fastest; every segment has seg_units
// numbers, of which those past the channel's last K-block stand for nothing.
struct Unit {
  long long u;      // global number
  int sb;           // subarray
  int G, c, seg;    // segment number in the subarray; channel, segment of it
  int slot;         // G % ring_slots
  unsigned gen;     // G / ring_slots
  int w, hb, k;     // unit in the segment
};

// Converter warps take their units in runs of p.run (1 or 2) consecutive units
// (of one segment: runs are of two only where its unit count is even): one slot claim and one
// publish (fence + release of the whole count) per run instead of per unit.
// Warp gw of nw takes runs gw, gw + nw, gw + 2 nw, ... of the global unit
// list.  Runs of one unit where there are too few units to go round.
constexpr int kUnitRun = 2;

// Unit u by division (a warp's first one, and the first in another subarray).
template <bool MULTI>
__device__ __forceinline__ void unit_locate(const Batch& bt, Unit& x) {
  x.sb = advance_sub<MULTI>(bt.unit_base, bt.nsub, x.u, x.sb);
  const Params& p = bt.sub[x.sb];
  const long long v = x.u - bt.unit_base[x.sb];
  x.G = static_cast<int>(v / p.seg_units);
  x.w = static_cast<int>(v - static_cast<long long>(x.G) * p.seg_units);
  x.gen = static_cast<unsigned>(x.G / p.ring_slots);
  x.slot = x.G - static_cast<int>(x.gen) * p.ring_slots;
}

// Next number of the warp; false at the end of the list.  The precomputed
// steps replace four divisions per unit: together with their dependent chains
// they were about a quarter of a converter warp's time per unit.
template <bool MULTI>
__device__ __forceinline__ bool unit_step(const Batch& bt, Unit& x, long long nw, long long total) {
  const int run = bt.sub[0].run;
  if ((x.u & (run - 1)) != run - 1) {
    ++x.u;
    ++x.w;
    return true;
  }
  x.u += 1 + (nw - 1) * run;
  if (x.u >= total) return false;
  if (MULTI && x.u >= bt.unit_base[x.sb + 1]) {
    unit_locate<MULTI>(bt, x);
    return true;
  }
  const Params& p = bt.sub[x.sb];
  x.w += p.step_rem - (run - 1);
  const int carry = x.w >= p.seg_units ? 1 : 0;
  x.w -= carry ? p.seg_units : 0;
  x.G += p.step_seg + carry;
  x.gen += static_cast<unsigned>(p.step_gen);
  x.slot += p.step_slot + carry;
  if (x.slot >= p.ring_slots) {
    x.slot -= p.ring_slots;
    ++x.gen;
  }
  return true;
}

// Channel, segment, half block and K-block of a number; false if it stands for
// nothing.
__device__ __forceinline__ bool unit_decode(const Params& p, Unit& x) {
  const bool last = x.G >= p.last_base;
  const int wv = last ? p.wave_full : fast_div(x.G, p.wave_segs, p.mag_wsegs);
  const int r = x.G - wv * p.wave_segs, width = last ? p.wave_last : p.wave;
  x.seg = fast_div(r, width, last ? p.mag_last : p.mag_wave);
  x.c = wv * p.wave + r - x.seg * width;
  x.hb = fast_div(x.w, p.seg_kb, p.mag_kb);
  x.k = x.w - x.hb * p.seg_kb;
  return x.seg * p.seg_kb + x.k < p.nkb;
}

template <bool MULTI>
__device__ __forceinline__ bool unit_first(const Batch& bt, Unit& x, long long gw, long long nw,
                                           long long total) {
  x.u = gw * bt.sub[0].run;
  x.sb = 0;
  if (x.u >= total) return false;
  unit_locate<MULTI>(bt, x);
  while (!unit_decode(bt.sub[x.sb], x))
    if (!unit_step<MULTI>(bt, x, nw, total)) return false;
  return true;
}
template <bool MULTI>
__device__ __forceinline__ bool unit_next(const Batch& bt, Unit& x, long long nw, long long total) {
  do {
    if (!unit_step<MULTI>(bt, x, nw, total)) return false;
  } while (!unit_decode(bt.sub[x.sb], x));
  return true;
}

// What unit x adds to its segment's ready counter: one, and for the last
// K-block of a half block in a short segment also its missing units, so that
// every segment counts seg_units.
__device__ __forceinline__ unsigned unit_weight(const Params& p, const Unit& x) {
  return x.seg * p.seg_kb + x.k == p.nkb - 1 ? static_cast<unsigned>(p.seg_kb - x.k) : 1u;
}

// Before a warp first writes segment G into its slot: the slot's previous
// segment (G - ring_slots) must have been read by all of its channel's items.
__device__ __forceinline__ bool claim_slot_warp(const Params& p, const Unit& x, int lane,
                                                volatile int* abort_flag) {
  bool ok = true;
  if (x.gen > 0 && lane == 0)
    ok = wait_counter(p.done + x.slot, x.gen * static_cast<unsigned>(p.ipc), p, abort_flag);
  // No proxy fence here: every bulk read of the slot's previous segment has
  // completed (its data sat in shared memory before the producer released
  // done[slot]), so the generic writes that follow cannot reach it.
  return __all_sync(0xffffffffu, ok);
}

// Would a claim of segment G's slot have to wait for the slot's previous
// segment?  (Checked before a warp waits while it holds an unpublished unit.)
__device__ __forceinline__ bool slot_busy(const Params& p, const Unit& x, int lane) {
  bool busy = false;
  if (x.gen > 0 && lane == 0)
    busy = ld_acquire(p.done + x.slot) < x.gen * static_cast<unsigned>(p.ipc);
  return __any_sync(0xffffffffu, busy);
}

// Publish one converted unit: every writing lane orders its generic stores
// before later async-proxy (bulk copy) reads, then one release.
__device__ __forceinline__ void publish_unit(const Params& p, int slot, int lane, unsigned n = 1) {
  if (p.test_no_publish) {  // failure-detection test: every consumer wait runs out
    __syncwarp();
    return;
  }
  fence_proxy_async_global();
  __syncwarp();
  if (lane == 0) red_release_add(p.ready + slot, n);
}

// Complex sample (re, im) of input a at sample t, channel c, as fp32.
template <int DT>
__device__ __forceinline__ float2 load_cx(const Params& p, int c, int a, int t) {
  const int64_t idx = (static_cast<int64_t>(t) * p.g.F + c) * p.n + a;
  if constexpr (DT == 1) {
    return __half22float2(static_cast<const __half2*>(p.in)[idx]);
  } else {
    return static_cast<const float2*>(p.in)[idx];
  }
}

// fp16x2 bits of (a, b).
__device__ __forceinline__ uint32_t h2bits(float a, float b) {
  __half2 q = __floats2half2_rn(a, b);
  return *reinterpret_cast<uint32_t*>(&q);
}
// fp16x2 bits of the residuals (a - fp16(a), b - fp16(b)) given h = fp16x2(a, b).
__device__ __forceinline__ uint32_t lo2bits(float a, float b, uint32_t h) {
  const __half2 hh = *reinterpret_cast<const __half2*>(&h);
  return h2bits(a - __low2float(hh), b - __high2float(hh));
}
// Four e4m3 bytes (a, b, c, d), a in the low byte, rounded to nearest with
// saturation to +-448.
__device__ __forceinline__ uint32_t e4m3x4(float a, float b, float c, float d) {
  const uint32_t lo = __nv_cvt_float2_to_fp8x2(make_float2(a, b), __NV_SATFINITE, __NV_E4M3);
  const uint32_t hi = __nv_cvt_float2_to_fp8x2(make_float2(c, d), __NV_SATFINITE, __NV_E4M3);
  return (lo & 0xffffu) | (hi << 16);
}

// Direct-load converter (float input of any row count), independent warps:
// lane l loads the complex samples of inputs l and l + 32 of the half block,
// 16 samples (32 loads) in flight at a time, applies the gains and the
// input's power-of-two scale (float input) and writes 16-byte chunks: per
// (input, plane) two fp16 chunks (8 samples each; HI/LO: two more into the
// L tile) or one e4m3 chunk (16 samples).
template <int DT, int FMT, bool MULTI, int SHAPE>
__device__ void converter_direct(const Batch& bt, int cw, int lane, volatile int* abort_flag) {
  static_assert(DT != 0, "8-bit input has its own converters");
  const long long total = table_end<MULTI>(bt.unit_base, bt.nsub);
  const long long nw = static_cast<long long>(gridDim.x) * conv_warps<FMT, DT>();
  int claimed = -1, claimed_sb = -1;
  Unit x;
  bool more = unit_first<MULTI>(bt, x, static_cast<long long>(blockIdx.x) * conv_warps<FMT, DT>() + cw, nw, total);
  for (; more; more = unit_next<MULTI>(bt, x, nw, total)) {
    const Params& p = bt.sub[x.sb];
    if (x.G != claimed || x.sb != claimed_sb) {
      if (!claim_slot_warp(p, x, lane, abort_flag)) return;
      claimed = x.G;
      claimed_sb = x.sb;
    }
    const int ib = x.hb >> 1;
    const int t0 = (x.seg * p.seg_kb + x.k) * kBK;  // first sample
    uint8_t* tre = ring_tile<FMT, SHAPE>(p, x.slot, 0, x.k, ib);
    uint8_t* tim = ring_tile<FMT, SHAPE>(p, x.slot, 1, x.k, ib);
    const int a0 = x.hb * 64 + lane, a1 = a0 + 32;
    const int row0 = (x.hb & 1) * 64 + lane;
    // y = g x 2^-e.
    float2 g0 = make_float2(1.f, 0.f), g1 = make_float2(1.f, 0.f);
    if (p.gains) {
      g0 = a0 < p.n ? p.gains[a0 % p.gain_n] : make_float2(0.f, 0.f);
      g1 = a1 < p.n ? p.gains[a1 % p.gain_n] : make_float2(0.f, 0.f);
    }
    if (p.in_amax) {
      const unsigned* am = p.in_amax + static_cast<int64_t>(x.c) * p.n;
      const float s0 = a0 < p.n ? exp2i(-scale_exp<FMT>(am[a0])) : 0.f;
      const float s1 = a1 < p.n ? exp2i(-scale_exp<FMT>(am[a1])) : 0.f;
      g0 = make_float2(g0.x * s0, g0.y * s0);  // exact: s is a power of two
      g1 = make_float2(g1.x * s1, g1.y * s1);
    }
    const bool apply = p.gains || p.in_amax;
#pragma unroll 1
    for (int g = 0; g < kUnitT / 16; ++g) {
      float2 v0[16], v1[16];
#pragma unroll
      for (int i = 0; i < 16; ++i) {
        const int t = t0 + g * 16 + i;
        v0[i] = (a0 < p.n && t < p.g.T) ? load_cx<DT>(p, x.c, a0, t) : make_float2(0.f, 0.f);
        v1[i] = (a1 < p.n && t < p.g.T) ? load_cx<DT>(p, x.c, a1, t) : make_float2(0.f, 0.f);
      }
      if (apply) {
#pragma unroll
        for (int i = 0; i < 16; ++i) {
          v0[i] = make_float2(g0.x * v0[i].x - g0.y * v0[i].y, g0.x * v0[i].y + g0.y * v0[i].x);
          v1[i] = make_float2(g1.x * v1[i].x - g1.y * v1[i].y, g1.x * v1[i].y + g1.y * v1[i].x);
        }
      }
      if constexpr (FMT == kFmtF8) {
        const uint32_t off = tile_off<FMT, SHAPE>(row0, g);
        const uint32_t off1 = tile_off<FMT, SHAPE>(row0 + 32, g);
        uint32_t r0[4], i0[4], r1[4], i1[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const float2* A = v0 + 4 * k;
          const float2* B = v1 + 4 * k;
          r0[k] = e4m3x4(A[0].x, A[1].x, A[2].x, A[3].x);
          i0[k] = e4m3x4(A[0].y, A[1].y, A[2].y, A[3].y);
          r1[k] = e4m3x4(B[0].x, B[1].x, B[2].x, B[3].x);
          i1[k] = e4m3x4(B[0].y, B[1].y, B[2].y, B[3].y);
        }
        *reinterpret_cast<uint4*>(tre + off) = make_uint4(r0[0], r0[1], r0[2], r0[3]);
        *reinterpret_cast<uint4*>(tim + off) = make_uint4(i0[0], i0[1], i0[2], i0[3]);
        *reinterpret_cast<uint4*>(tre + off1) = make_uint4(r1[0], r1[1], r1[2], r1[3]);
        *reinterpret_cast<uint4*>(tim + off1) = make_uint4(i1[0], i1[1], i1[2], i1[3]);
      } else {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const uint32_t off = tile_off<FMT, SHAPE>(row0, 2 * g + h);
          const uint32_t off1 = tile_off<FMT, SHAPE>(row0 + 32, 2 * g + h);
          uint32_t r0[4], i0[4], r1[4], i1[4];
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            const float2 a = v0[8 * h + 2 * k], b = v0[8 * h + 2 * k + 1];
            const float2 c = v1[8 * h + 2 * k], d = v1[8 * h + 2 * k + 1];
            r0[k] = h2bits(a.x, b.x);
            i0[k] = h2bits(a.y, b.y);
            r1[k] = h2bits(c.x, d.x);
            i1[k] = h2bits(c.y, d.y);
          }
          *reinterpret_cast<uint4*>(tre + off) = make_uint4(r0[0], r0[1], r0[2], r0[3]);
          *reinterpret_cast<uint4*>(tim + off) = make_uint4(i0[0], i0[1], i0[2], i0[3]);
          *reinterpret_cast<uint4*>(tre + off1) = make_uint4(r1[0], r1[1], r1[2], r1[3]);
          *reinterpret_cast<uint4*>(tim + off1) = make_uint4(i1[0], i1[1], i1[2], i1[3]);
          if constexpr (FMT == kFmtHiLo) {
            // Residual tile of the same K-block: K-tile seg_kb + k.
            const int64_t lo_off = static_cast<int64_t>(p.seg_kb) * p.nib * FmtT<FMT, SHAPE>::kKbBytes;
            uint32_t l0[4], m0[4], l1[4], m1[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
              const float2 a = v0[8 * h + 2 * k], b = v0[8 * h + 2 * k + 1];
              const float2 c = v1[8 * h + 2 * k], d = v1[8 * h + 2 * k + 1];
              l0[k] = lo2bits(a.x, b.x, r0[k]);
              m0[k] = lo2bits(a.y, b.y, i0[k]);
              l1[k] = lo2bits(c.x, d.x, r1[k]);
              m1[k] = lo2bits(c.y, d.y, i1[k]);
            }
            *reinterpret_cast<uint4*>(tre + lo_off + off) = make_uint4(l0[0], l0[1], l0[2], l0[3]);
            *reinterpret_cast<uint4*>(tim + lo_off + off) = make_uint4(m0[0], m0[1], m0[2], m0[3]);
            *reinterpret_cast<uint4*>(tre + lo_off + off1) = make_uint4(l1[0], l1[1], l1[2], l1[3]);
            *reinterpret_cast<uint4*>(tim + lo_off + off1) = make_uint4(m1[0], m1[1], m1[2], m1[3]);
          }
        }
      }
    }
    publish_unit(p, x.slot, lane, unit_weight(p, x));
    if (*abort_flag) return;
  }
}

// Bounded wait for the warp's TMA box still in flight (completing phase
// `phase` of `bar`): a converter that gives up never leaves a copy landing in
// shared memory after it has returned.
__device__ __forceinline__ void drain_tma(uint32_t bar, uint32_t phase, bool pending,
                                          unsigned long long timeout_ns) {
  if (pending) {
    const uint64_t t0 = ptx::globaltimer();
    while (!ptx::mbar_try_wait(bar, phase) && ptx::globaltimer() - t0 < timeout_ns) {
    }
  }
  __syncwarp();
}

// 8-bit words to operands.  A word is (re, im) of a lane's two inputs, tile rows
// 2l and 2l + 1, at one sample; the words of a 16-byte chunk (8 samples in fp16,
// 16 in e4m3) make 32 contiguous bytes of a plane, so a warp store covers 1 KiB.
// fp16, one plane (j: 0 re, 1 im), with the largest |x| of each half of `mq`.
__device__ __forceinline__ void store_rows_f16(uint8_t* dst, const uint32_t* W, uint32_t j, __half2& mq, uint64_t pol) {
  uint32_t v[8];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    v[k] = pair_i8(W[2 * k], W[2 * k + 1], j);
    v[4 + k] = pair_i8(W[2 * k], W[2 * k + 1], j + 2);
  }
#pragma unroll
  for (int k = 0; k < 8; k += 2)
    mq = __hmax2(mq, __hmax2(__habs2(*reinterpret_cast<const __half2*>(&v[k])),
                             __habs2(*reinterpret_cast<const __half2*>(&v[k + 1]))));
  ptx::st_global_v8_hint(dst, v, pol);
}
// Component j of four consecutive samples as four e4m3 bytes: the exact fp16
// pair conversion, then one fp16x2 -> e4m3x2 conversion per pair (exact for
// |x| <= 16).
__device__ __forceinline__ uint32_t quad_f8(const uint32_t* W, uint32_t j) {
  const uint32_t h01 = pair_i8(W[0], W[1], j), h23 = pair_i8(W[2], W[3], j);
  __half2_raw r01, r23;
  r01.x = static_cast<unsigned short>(h01 & 0xffffu);
  r01.y = static_cast<unsigned short>(h01 >> 16);
  r23.x = static_cast<unsigned short>(h23 & 0xffffu);
  r23.y = static_cast<unsigned short>(h23 >> 16);
  const uint32_t e01 = __nv_cvt_halfraw2_to_fp8x2(r01, __NV_SATFINITE, __NV_E4M3);
  const uint32_t e23 = __nv_cvt_halfraw2_to_fp8x2(r23, __NV_SATFINITE, __NV_E4M3);
  return (e01 & 0xffffu) | (e23 << 16);
}
// e4m3, both planes, with the largest |x| of each byte of `mb`.
__device__ __forceinline__ void store_rows_f8(uint8_t* re, uint8_t* im, const uint32_t* W, uint32_t& mb,
                                              uint64_t pol) {
#pragma unroll
  for (int t = 0; t < 16; ++t) mb = __vmaxu4(mb, __vabs4(W[t]));
  uint32_t vr[8], vi[8];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    vr[k] = quad_f8(W + 4 * k, 0);
    vi[k] = quad_f8(W + 4 * k, 1);
    vr[4 + k] = quad_f8(W + 4 * k, 2);
    vi[4 + k] = quad_f8(W + 4 * k, 3);
  }
  ptx::st_global_v8_hint(re, vr, pol);
  ptx::st_global_v8_hint(im, vi, pol);
}

// 8-bit converter with TMA-staged input.  Each converter warp is an
// independent worker on its own stream of units (u = global warp id + k *
// warps, channel-major), with an 8 KiB staging buffer ([64 samples][128
// rows] int8 = 64 inputs x {re, im}) that always holds its next unit's box
// in flight while the current one is converted.  A warp claims a slot for
// itself and publishes each unit on its own: no barrier couples the warps.
// A unit is published after the next unit's shared-memory reads, so its
// stores have drained by the time the proxy fence waits for them; a warp
// that would have to wait for a slot publishes first (a consumer of the
// slot's previous channel may need that unit).
template <int FMT, bool MULTI, int SHAPE>
__device__ void converter_tma(const Batch& bt, uint32_t buf, uint32_t bar, int cw, int lane,
                              volatile int* abort_flag) {
  static_assert(FMT == kFmtF16 || FMT == kFmtF8, "8-bit input: fp16 or e4m3 operands");
  const long long total = table_end<MULTI>(bt.unit_base, bt.nsub);
  const long long nw = static_cast<long long>(gridDim.x) * conv_warps<FMT, 0>();
  const ptx::WaitCtl wc{bt.sub[0].timeout_ns, bt.sub[0].status, abort_flag};
  bool tma_pending = false;  // a box issued and not yet waited for
  auto issue = [&](const Unit& x) {
    tma_pending = true;
    if (lane == 0) {
      ptx::mbar_arrive_expect_tx(bar, kConvBufBytes);
      // The input streams through once: first in line for L2 replacement, so
      // the operand ring it is converted into stays resident.
      ptx::tma_load_3d_hint(buf, &bt.maps[x.sb], bar, x.hb * kUnitRows, x.c,
                            (x.seg * bt.sub[x.sb].seg_kb + x.k) * kUnitT, ptx::l2_policy_evict_first());
    }
  };
  const uint32_t* src = reinterpret_cast<const uint32_t*>(__cvta_shared_to_generic(static_cast<size_t>(buf)));
  // Lane l converts inputs 2l and 2l + 1 of the half block: word l of each
  // 128-byte sample row holds (re, im) of both.  Per 8-sample chunk and plane
  // the lane writes tile rows 2l and 2l + 1 (32 contiguous bytes), so a warp
  // store covers 1 KiB.
  uint32_t phase = 0;
  int claimed = -1, claimed_sb = -1;
  // Converted units of a run not yet published: their subarray, slot, run, count.
  const Params* pend = nullptr;
  int pend_slot = 0;
  long long pend_run = -1;
  unsigned pend_n = 0;
  Unit x;
  bool more = unit_first<MULTI>(bt, x, static_cast<long long>(blockIdx.x) * conv_warps<FMT, 0>() + cw, nw, total);
  if (more) issue(x);
  while (more) {
    const Params& p = bt.sub[x.sb];
    if (x.G != claimed || x.sb != claimed_sb) {
      if (pend && slot_busy(p, x, lane)) {
        publish_unit(*pend, pend_slot, lane, pend_n);
        pend = nullptr;
      }
      if (!claim_slot_warp(p, x, lane, abort_flag)) {
        drain_tma(bar, phase, tma_pending, wc.timeout_ns);
        return;
      }
      claimed = x.G;
      claimed_sb = x.sb;
    }
    const bool got = ptx::wait_bounded(bar, phase, wc);
    if (!__all_sync(0xffffffffu, got)) {
      drain_tma(bar, phase, tma_pending, wc.timeout_ns);
      return;
    }
    tma_pending = false;
    phase ^= 1u;
    // Both inputs' kUnitT samples into registers, then refill the buffer.
    uint32_t w[kUnitT];
#pragma unroll
    for (int t = 0; t < kUnitT; ++t) w[t] = src[t * (kUnitRows / 4) + lane];
    __syncwarp();
    ptx::fence_proxy_async_smem();
    Unit nx = x;
    more = unit_next<MULTI>(bt, nx, nw, total);
    if (more) issue(nx);
    // A finished run is published now: its stores have drained during this
    // unit's shared-memory reads.
    if (pend && pend_run != x.u / p.run) {
      publish_unit(*pend, pend_slot, lane, pend_n);
      pend = nullptr;
    }
    const int ib = x.hb >> 1;
    uint8_t* tre = ring_tile<FMT, SHAPE>(p, x.slot, 0, x.k, ib);
    uint8_t* tim = ring_tile<FMT, SHAPE>(p, x.slot, 1, x.k, ib);
    const int row = (x.hb & 1) * 64 + 2 * lane;  // tile rows 2l and 2l + 1
    // Ring tiles are read back by every block of the channel: keep them in L2.
    const uint64_t pol_last = ptx::l2_policy_evict_last();
    unsigned m = 0;  // max |x| over the unit (zero-filled rows and samples contribute 0)
    if constexpr (FMT == kFmtF16) {
      // max |x| from the converted (exact) fp16 values.
      __half2 mx[2];
#pragma unroll
      for (int q = 0; q < 2; ++q) mx[q] = __float2half2_rn(0.f);
#pragma unroll
      for (int cc = 0; cc < kUnitT / 8; ++cc) {
        const uint32_t off = tile_off<FMT, SHAPE>(row, cc);
        store_rows_f16(tre + off, w + 8 * cc, 0u, mx[0], pol_last);
        store_rows_f16(tim + off, w + 8 * cc, 1u, mx[1], pol_last);
      }
      const __half2 mm = __hmax2(mx[0], mx[1]);
      m = static_cast<unsigned>(fmaxf(__low2float(mm), __high2float(mm)));
    } else {
      // e4m3 operands: exact for |x| <= 16 (a larger value sets the range
      // status bit below).  16-sample chunks; rows 2l and 2l + 1 per store.
      uint32_t mb = 0;  // per-byte |x| maximum
#pragma unroll
      for (int cc = 0; cc < kUnitT / 16; ++cc) {
        const uint32_t off = tile_off<FMT, SHAPE>(row, cc);
        store_rows_f8(tre + off, tim + off, w + 16 * cc, mb, pol_last);
      }
      m = max(max(mb & 0xffu, (mb >> 8) & 0xffu), max((mb >> 16) & 0xffu, mb >> 24));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
    if (lane == 0) {
      atomicMax(p.amax + x.G, m);
      if (FMT == kFmtF8 && m > 16) atomicOr(p.status, kStatusRange);
    }
    if (!pend) {
      pend = &p;
      pend_slot = x.slot;
      pend_run = x.u / p.run;
      pend_n = 0;
    }
    pend_n += unit_weight(p, x);
    x = nx;
    if (*abort_flag) {
      drain_tma(bar, phase, tma_pending, wc.timeout_ns);
      return;
    }
  }
  if (pend) publish_unit(*pend, pend_slot, lane, pend_n);
}

// 8-bit converter for rows that TMA cannot stride (not a multiple of 16 bytes).
// As converter_tma, but the words are loaded straight into registers: an even
// number of inputs (EVEN) has its rows on 4 bytes, an odd one is read in
// 16-bit halves that are joined when they are used.  As soon as 8 samples are
// converted their registers take the loads kRing chunks on (64 samples, or
// 32), which so have that long to arrive.  (On rows that TMA can stride this is
// the slower one: 256 stations x 2 pols, F=1024, T=1000 1.16 against 1.03 ms.)
// Measured against converting single components by way of floats, for any row:
// 37 stations x 2 pols, F=2048, T=1000 1741 -> 440 us; 131 stations x 1 pol,
// F=300, T=500 271 -> 140 us.
// A warp publishes each run at the start of the run after it; a warp that would
// have to wait for a slot publishes first (a consumer of the slot's previous
// segment may need that run).
template <int FMT, bool MULTI, int SHAPE, bool EVEN>
__device__ void converter_words(const Batch& bt, int cw, int lane, volatile int* abort_flag) {
  static_assert(FMT == kFmtF16 || FMT == kFmtF8, "8-bit input: fp16 or e4m3 operands");
  const long long total = table_end<MULTI>(bt.unit_base, bt.nsub);
  const long long nw = static_cast<long long>(gridDim.x) * conv_warps<FMT, 0>();
  // The input streams through once: first in line for L2 replacement, so the
  // operand ring it is converted into stays resident.  Ring tiles are read
  // back by every block of the channel: keep them in L2.
  const uint64_t pol_first = ptx::l2_policy_evict_first(), pol_last = ptx::l2_policy_evict_last();
  // Where a unit's words come from: this lane's word of sample 0, the bytes
  // from sample to sample, and the samples to load (0: no such input).
  struct Src {
    const uint8_t* ptr;
    int64_t step;
    int count, count_hi;  // of the word's first and second input
  };
  const uint32_t lane4 = static_cast<uint32_t>(lane) * 4u;
  auto source = [&](const Unit& x) {
    const Params& p = bt.sub[x.sb];
    const int t0 = (x.seg * p.seg_kb + x.k) * kBK;
    Src s;
    s.step = static_cast<int64_t>(p.g.F) * p.g.R;
    s.ptr = static_cast<const uint8_t*>(p.in) + t0 * s.step + static_cast<int64_t>(x.c) * p.g.R +
            x.hb * kUnitRows;
    const int ns = min(kBK, p.g.T - t0), row = x.hb * kUnitRows + static_cast<int>(lane4);
    s.count = row < p.g.R ? ns : 0;
    s.count_hi = row + 2 < p.g.R ? ns : 0;
    return s;
  };
  // The registers: a ring of 8-sample chunks, one word per sample or two halves.
  constexpr int kRing = EVEN ? 8 : 4, kPer = EVEN ? 8 : 16;
  uint32_t w[kRing * kPer];
  // Chunk cc of a unit into its registers (zero past the end).
  auto load8 = [&](const Src& s, int cc) {
    uint32_t* r = w + cc % kRing * kPer;
    const uint8_t* q = s.ptr + 8 * cc * s.step + lane4;
#pragma unroll
    for (int t = 0; t < 8; ++t) {
      if constexpr (EVEN) {
        r[t] = ptx::ld_global_b32_if(q + t * s.step, pol_first, 8 * cc + t < s.count);
      } else {
        r[t] = ptx::ld_global_u16_if(q + t * s.step, pol_first, 8 * cc + t < s.count);
        r[8 + t] = ptx::ld_global_u16_if(q + t * s.step + 2, pol_first, 8 * cc + t < s.count_hi);
      }
    }
  };
  // Chunk cc's words.
  auto words8 = [&](int cc, uint32_t* W) {
    const uint32_t* r = w + cc % kRing * kPer;
#pragma unroll
    for (int t = 0; t < 8; ++t) W[t] = EVEN ? r[t] : (r[t] | r[8 + t] << 16);
  };
  int claimed = -1, claimed_sb = -1;
  // Converted units of a run not yet published: their subarray, slot, run, count.
  const Params* pend = nullptr;
  int pend_slot = 0;
  long long pend_run = -1;
  unsigned pend_n = 0;
  Unit x;
  bool more = unit_first<MULTI>(bt, x, static_cast<long long>(blockIdx.x) * conv_warps<FMT, 0>() + cw, nw, total);
  Src cs = {nullptr, 0, 0, 0};
  if (more) {
    cs = source(x);
#pragma unroll
    for (int cc = 0; cc < kRing; ++cc) load8(cs, cc);
  }
  while (more) {
    const Params& p = bt.sub[x.sb];
    if (x.G != claimed || x.sb != claimed_sb) {
      if (pend && slot_busy(p, x, lane)) {
        publish_unit(*pend, pend_slot, lane, pend_n);
        pend = nullptr;
      }
      if (!claim_slot_warp(p, x, lane, abort_flag)) return;
      claimed = x.G;
      claimed_sb = x.sb;
    }
    Unit nx = x;
    more = unit_next<MULTI>(bt, nx, nw, total);
    Src ns = {nullptr, 0, 0, 0};
    if (more) ns = source(nx);
    // The chunk that takes chunk cc's registers: of this unit or the next.
    auto reload = [&](int cc) {
      if (cc + kRing < kBK / 8)
        load8(cs, cc + kRing);
      else
        load8(ns, cc + kRing - kBK / 8);
    };
    const int ib = x.hb >> 1;
    uint8_t* tre = ring_tile<FMT, SHAPE>(p, x.slot, 0, x.k, ib);
    uint8_t* tim = ring_tile<FMT, SHAPE>(p, x.slot, 1, x.k, ib);
    const int row = (x.hb & 1) * 64 + 2 * lane;  // tile rows 2l and 2l + 1
    // A finished run is published now: its last stores have had some time.
    if (pend && pend_run != x.u / p.run) {
      publish_unit(*pend, pend_slot, lane, pend_n);
      pend = nullptr;
    }
    unsigned m = 0;  // max |x| over the unit (rows and samples past the end contribute 0)
    if constexpr (FMT == kFmtF16) {
      // max |x| from the converted (exact) fp16 values.
      __half2 mx[2];
#pragma unroll
      for (int q = 0; q < 2; ++q) mx[q] = __float2half2_rn(0.f);
#pragma unroll
      for (int cc = 0; cc < kBK / 8; ++cc) {
        const uint32_t off = tile_off<FMT, SHAPE>(row, cc);
        uint32_t W[8];
        words8(cc, W);
        store_rows_f16(tre + off, W, 0u, mx[0], pol_last);
        store_rows_f16(tim + off, W, 1u, mx[1], pol_last);
        reload(cc);
      }
      const __half2 mm = __hmax2(mx[0], mx[1]);
      m = static_cast<unsigned>(fmaxf(__low2float(mm), __high2float(mm)));
    } else {
      // e4m3 operands: exact for |x| <= 16 (a larger value sets the range
      // status bit below).  16-sample chunks; rows 2l and 2l + 1 per store.
      uint32_t mb = 0;  // per-byte |x| maximum
#pragma unroll
      for (int cc = 0; cc < kBK / 16; ++cc) {
        const uint32_t off = tile_off<FMT, SHAPE>(row, cc);
        uint32_t W[16];
        words8(2 * cc, W);
        words8(2 * cc + 1, W + 8);
        store_rows_f8(tre + off, tim + off, W, mb, pol_last);
        reload(2 * cc);
        reload(2 * cc + 1);
      }
      m = max(max(mb & 0xffu, (mb >> 8) & 0xffu), max((mb >> 16) & 0xffu, mb >> 24));
    }
    m = __reduce_max_sync(0xffffffffu, m);
    if (lane == 0) {
      atomicMax(p.amax + x.G, m);
      if (FMT == kFmtF8 && m > 16) atomicOr(p.status, kStatusRange);
    }
    if (!pend) {
      pend = &p;
      pend_slot = x.slot;
      pend_run = x.u / p.run;
      pend_n = 0;
    }
    pend_n += unit_weight(p, x);
    x = nx;
    cs = ns;
    if (*abort_flag) return;
  }
  if (pend) publish_unit(*pend, pend_slot, lane, pend_n);
}

// Convert 16 samples of two inputs (v0: input a0, v1: input a1 = a0 + 32;
// gains and scale already applied) into the tiles of one K-block: fp16 (two
// 8-sample chunks from chunk8), hi/lo (the same in the H tiles plus the
// residuals in the L tiles) or e4m3 (one 16-sample chunk).
template <int FMT, int SHAPE>
__device__ __forceinline__ void store_group16(const Params& p, uint8_t* tre, uint8_t* tim, int row0,
                                              int chunk8, const float2 (&v0)[16],
                                              const float2 (&v1)[16], uint64_t pol) {
  auto st = [&](uint8_t* dst, uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
    ptx::st_global_v4_hint(dst, a, b, c, d, pol);
  };
  if constexpr (FMT == kFmtF8) {
    const uint32_t off = tile_off<FMT, SHAPE>(row0, chunk8 / 2);
    const uint32_t off1 = tile_off<FMT, SHAPE>(row0 + 32, chunk8 / 2);
    uint32_t r0[4], i0[4], r1[4], i1[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const float2* A = v0 + 4 * k;
      const float2* B = v1 + 4 * k;
      r0[k] = e4m3x4(A[0].x, A[1].x, A[2].x, A[3].x);
      i0[k] = e4m3x4(A[0].y, A[1].y, A[2].y, A[3].y);
      r1[k] = e4m3x4(B[0].x, B[1].x, B[2].x, B[3].x);
      i1[k] = e4m3x4(B[0].y, B[1].y, B[2].y, B[3].y);
    }
    st(tre + off, r0[0], r0[1], r0[2], r0[3]);
    st(tim + off, i0[0], i0[1], i0[2], i0[3]);
    st(tre + off1, r1[0], r1[1], r1[2], r1[3]);
    st(tim + off1, i1[0], i1[1], i1[2], i1[3]);
  } else {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const uint32_t off = tile_off<FMT, SHAPE>(row0, chunk8 + h);
      const uint32_t off1 = tile_off<FMT, SHAPE>(row0 + 32, chunk8 + h);
      uint32_t r0[4], i0[4], r1[4], i1[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const float2 a = v0[8 * h + 2 * k], b = v0[8 * h + 2 * k + 1];
        const float2 c = v1[8 * h + 2 * k], d = v1[8 * h + 2 * k + 1];
        r0[k] = h2bits(a.x, b.x);
        i0[k] = h2bits(a.y, b.y);
        r1[k] = h2bits(c.x, d.x);
        i1[k] = h2bits(c.y, d.y);
      }
      st(tre + off, r0[0], r0[1], r0[2], r0[3]);
      st(tim + off, i0[0], i0[1], i0[2], i0[3]);
      st(tre + off1, r1[0], r1[1], r1[2], r1[3]);
      st(tim + off1, i1[0], i1[1], i1[2], i1[3]);
      if constexpr (FMT == kFmtHiLo) {
        // Residual tile of the same K-block: K-tile seg_kb + k.
        const int64_t lo_off = static_cast<int64_t>(p.seg_kb) * p.nib * FmtT<FMT, SHAPE>::kKbBytes;
        uint32_t l0[4], m0[4], l1[4], m1[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const float2 a = v0[8 * h + 2 * k], b = v0[8 * h + 2 * k + 1];
          const float2 c = v1[8 * h + 2 * k], d = v1[8 * h + 2 * k + 1];
          l0[k] = lo2bits(a.x, b.x, r0[k]);
          m0[k] = lo2bits(a.y, b.y, i0[k]);
          l1[k] = lo2bits(c.x, d.x, r1[k]);
          m1[k] = lo2bits(c.y, d.y, i1[k]);
        }
        st(tre + lo_off + off, l0[0], l0[1], l0[2], l0[3]);
        st(tim + lo_off + off, m0[0], m0[1], m0[2], m0[3]);
        st(tre + lo_off + off1, l1[0], l1[1], l1[2], l1[3]);
        st(tim + lo_off + off1, m1[0], m1[1], m1[2], m1[3]);
      }
    }
  }
}

// Float converter with TMA-staged input: boxes of 64 inputs x kFBox samples
// (8 KiB: complex fp16, 32 samples, or complex fp32, 16 samples) pass
// through the warp's one staging buffer, kUnitT / kFBox boxes per unit;
// while one box is converted the next (of this unit or of the next) is in
// flight.  Units are taken in runs and published as in converter_tma.
template <int DT, int FMT, bool MULTI, int SHAPE>
__device__ void converter_tma_float(const Batch& bt, uint32_t buf, uint32_t bar, int cw, int lane,
                                    volatile int* abort_flag) {
  constexpr int kCx = DT == 1 ? 4 : 8;  // bytes per complex sample
  constexpr int kFBox = kConvBufBytes / (64 * kCx);
  constexpr int kBoxes = kUnitT / kFBox;
  static_assert(kFBox % 16 == 0 && kUnitT % kFBox == 0, "boxes hold whole 16-sample groups");
  const long long total = table_end<MULTI>(bt.unit_base, bt.nsub);
  const long long nw = static_cast<long long>(gridDim.x) * conv_warps<FMT, DT>();
  const ptx::WaitCtl wc{bt.sub[0].timeout_ns, bt.sub[0].status, abort_flag};
  bool tma_pending = false;  // a box issued and not yet waited for
  auto issue = [&](const Unit& x, int j) {
    tma_pending = true;
    if (lane == 0) {
      ptx::mbar_arrive_expect_tx(bar, kConvBufBytes);
      // Map elements: one complex fp16 (32-bit) or one fp32 component.
      const int ex = DT == 1 ? x.hb * 64 : x.hb * 128;
      ptx::tma_load_3d_hint(buf, &bt.maps[x.sb], bar, ex, x.c,
                            (x.seg * bt.sub[x.sb].seg_kb + x.k) * kUnitT + j * kFBox,
                            ptx::l2_policy_evict_first());
    }
  };
  const uint8_t* src = reinterpret_cast<const uint8_t*>(__cvta_shared_to_generic(static_cast<size_t>(buf)));
  const uint64_t pol_last = ptx::l2_policy_evict_last();
  uint32_t phase = 0;
  int claimed = -1, claimed_sb = -1;
  // Converted units of a run not yet published: their subarray, slot, run, count.
  const Params* pend = nullptr;
  int pend_slot = 0;
  long long pend_run = -1;
  unsigned pend_n = 0;
  Unit x;
  bool more = unit_first<MULTI>(bt, x, static_cast<long long>(blockIdx.x) * conv_warps<FMT, DT>() + cw, nw, total);
  if (more) issue(x, 0);
  while (more) {
    const Params& p = bt.sub[x.sb];
    if (x.G != claimed || x.sb != claimed_sb) {
      if (pend && slot_busy(p, x, lane)) {
        publish_unit(*pend, pend_slot, lane, pend_n);
        pend = nullptr;
      }
      if (!claim_slot_warp(p, x, lane, abort_flag)) {
        drain_tma(bar, phase, tma_pending, wc.timeout_ns);
        return;
      }
      claimed = x.G;
      claimed_sb = x.sb;
    }
    const int ib = x.hb >> 1;
    uint8_t* tre = ring_tile<FMT, SHAPE>(p, x.slot, 0, x.k, ib);
    uint8_t* tim = ring_tile<FMT, SHAPE>(p, x.slot, 1, x.k, ib);
    const int a0 = x.hb * 64 + lane, a1 = a0 + 32;
    const int row0 = (x.hb & 1) * 64 + lane;
    Unit nx = x;
    more = unit_next<MULTI>(bt, nx, nw, total);
    // y = g x 2^-e.
    float2 g0 = make_float2(1.f, 0.f), g1 = make_float2(1.f, 0.f);
    if (p.gains) {
      g0 = a0 < p.n ? p.gains[a0 % p.gain_n] : make_float2(0.f, 0.f);
      g1 = a1 < p.n ? p.gains[a1 % p.gain_n] : make_float2(0.f, 0.f);
    }
    if (p.in_amax) {
      const unsigned* am = p.in_amax + static_cast<int64_t>(x.c) * p.n;
      const float s0 = a0 < p.n ? exp2i(-scale_exp<FMT>(am[a0])) : 0.f;
      const float s1 = a1 < p.n ? exp2i(-scale_exp<FMT>(am[a1])) : 0.f;
      g0 = make_float2(g0.x * s0, g0.y * s0);  // exact: s is a power of two
      g1 = make_float2(g1.x * s1, g1.y * s1);
    }
#pragma unroll 1
    for (int j = 0; j < kBoxes; ++j) {
      const bool got = ptx::wait_bounded(bar, phase, wc);
      if (!__all_sync(0xffffffffu, got)) {
        drain_tma(bar, phase, tma_pending, wc.timeout_ns);
        return;
      }
      tma_pending = false;
      phase ^= 1u;
      // Lane l: inputs l and l + 32 of the box's 64, every sample.
      using Raw = typename std::conditional<DT == 1, uint32_t, float2>::type;
      const Raw* box = reinterpret_cast<const Raw*>(src);
      Raw w0[kFBox], w1[kFBox];
#pragma unroll
      for (int t = 0; t < kFBox; ++t) {
        w0[t] = box[t * 64 + lane];
        w1[t] = box[t * 64 + 32 + lane];
      }
      __syncwarp();
      ptx::fence_proxy_async_smem();
      if (j + 1 < kBoxes) {
        issue(x, j + 1);
      } else if (more) {
        issue(nx, 0);
      }
      if (j == 0 && pend && pend_run != x.u / p.run) {
        publish_unit(*pend, pend_slot, lane, pend_n);
        pend = nullptr;
      }
#pragma unroll
      for (int g16 = 0; g16 < kFBox / 16; ++g16) {
        float2 v0[16], v1[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) {
          float2 c0, c1;
          if constexpr (DT == 1) {
            c0 = __half22float2(*reinterpret_cast<const __half2*>(&w0[16 * g16 + i]));
            c1 = __half22float2(*reinterpret_cast<const __half2*>(&w1[16 * g16 + i]));
          } else {
            c0 = w0[16 * g16 + i];
            c1 = w1[16 * g16 + i];
          }
          v0[i] = make_float2(g0.x * c0.x - g0.y * c0.y, g0.x * c0.y + g0.y * c0.x);
          v1[i] = make_float2(g1.x * c1.x - g1.y * c1.y, g1.x * c1.y + g1.y * c1.x);
        }
        store_group16<FMT, SHAPE>(p, tre, tim, row0, (j * kFBox + 16 * g16) / 8, v0, v1, pol_last);
      }
    }
    if (!pend) {
      pend = &p;
      pend_slot = x.slot;
      pend_run = x.u / p.run;
      pend_n = 0;
    }
    pend_n += unit_weight(p, x);
    x = nx;
    if (*abort_flag) {
      drain_tma(bar, phase, tma_pending, wc.timeout_ns);
      return;
    }
  }
  if (pend) publish_unit(*pend, pend_slot, lane, pend_n);
}

// --------------------------------------------------------------- epilogue

// How a piece's fp32 sums become the stored words: as they are (float input)
// or int32 (8-bit input).
enum : int { kWordFloat = 0, kWordInt = 1 };
template <int WORD>
__device__ __forceinline__ uint32_t out_word(uint32_t u) {
  if constexpr (WORD == kWordFloat) return u;
  return static_cast<uint32_t>(__float2int_rn(__uint_as_float(u)));
}

// Store one 32-column piece: values v_re[j], v_im[j] of V(a, b0 + j).
template <int WORD>
__device__ __forceinline__ void store_piece(const uint32_t (&re)[32], const uint32_t (&im)[32],
                                            const Params& p, int f, int a, int b0, bool add, uint64_t pol) {
  constexpr bool IS_INT = WORD != kWordFloat;
  using T = typename std::conditional<IS_INT, int, float>::type;
  const Geometry& g = p.g;
  T* out = static_cast<T*>(p.out);
  auto val = [&](uint32_t u) -> T {
    if constexpr (IS_INT) {
      return static_cast<int>(out_word<WORD>(u));
    } else {
      return __uint_as_float(u);
    }
  };
  // Two polarisations, overwrite, 32-byte aligned output: the lanes of a
  // station's two rows (a, a ^ 1; both valid or both not, n being even)
  // exchange halves so that each writes whole 32-byte baseline records.
  const bool pairs = g.P == 2 && !add && (reinterpret_cast<uintptr_t>(out) & 31) == 0;
  const bool valid = a < p.n;
  if (!valid && !pairs) return;
  // Real channel, row station and first column station (packed channels:
  // columns of another channel of the pack fall outside 0 <= s2 <= s1).
  int fr = f, s1 = a >> (g.P - 1), s2_0 = b0 >> (g.P - 1);  // P is 1 or 2
  if (p.pack > 1) {
    const int j = s1 / p.Nr;
    s1 -= j * p.Nr;
    s2_0 -= j * p.Nr;
    fr = f * p.pack + j;
  }
  const int64_t krow = static_cast<int64_t>(fr) * p.NBr + static_cast<int64_t>(s1) * (s1 + 1) / 2;
  if (pairs) {
    const int p1 = a & 1;
    uint32_t* o8 = reinterpret_cast<uint32_t*>(out + krow * 8);  // record of s2 at o8 + 8 s2
#pragma unroll
    for (int m = 0; m < 8; ++m) {
      // This lane's products for column stations 2m (A) and 2m + 1 (B) of the piece.
      uint32_t A[4], B[4], rec[8];
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        A[2 * q] = out_word<WORD>(re[4 * m + q]);
        A[2 * q + 1] = out_word<WORD>(im[4 * m + q]);
        B[2 * q] = out_word<WORD>(re[4 * m + 2 + q]);
        B[2 * q + 1] = out_word<WORD>(im[4 * m + 2 + q]);
      }
      // Row p1 = 0 writes baseline 2m, row p1 = 1 baseline 2m + 1; each sends
      // the partner the half it needs.
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const uint32_t got = __shfl_xor_sync(0xffffffffu, p1 ? A[k] : B[k], 1);
        rec[k] = p1 ? got : A[k];
        rec[4 + k] = p1 ? B[k] : got;
      }
      const int s2 = s2_0 + 2 * m + p1;
      if (valid && s2 >= 0 && s2 <= s1)
        ptx::st_global_v8_hint(o8 + 8 * static_cast<int64_t>(s2), rec, pol);
    }
  } else if (g.P == 2) {
    const int p1 = a & 1;
    using V4 = typename std::conditional<IS_INT, int4, float4>::type;
    V4* o4 = reinterpret_cast<V4*>(out + (krow * 4 + p1 * 2) * 2);  // (p1,0),(p1,1) of s2 at o4[2 s2]
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      V4 old[8];
      if (add) {
        // Loads of a half first: independent of the stores that follow.
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const int s2 = s2_0 + 8 * h + j;
          if (s2 >= 0 && s2 <= s1) old[j] = o4[2 * s2];
        }
      }
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const int jj = 8 * h + j;
        const int s2 = s2_0 + jj;
        if (s2 >= 0 && s2 <= s1) {
          V4 v;
          v.x = val(re[2 * jj]);
          v.y = val(im[2 * jj]);
          v.z = val(re[2 * jj + 1]);
          v.w = val(im[2 * jj + 1]);
          if (add) {
            v.x += old[j].x;
            v.y += old[j].y;
            v.z += old[j].z;
            v.w += old[j].w;
          }
          o4[2 * s2] = v;
        }
      }
    }
  } else {
    using V2 = typename std::conditional<IS_INT, int2, float2>::type;
    V2* o2 = reinterpret_cast<V2*>(out + krow * 2);  // baseline s2 at o2[s2]
#pragma unroll
    for (int h = 0; h < 4; ++h) {
      V2 old[8];
      if (add) {
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const int s2 = s2_0 + 8 * h + j;
          if (s2 >= 0 && s2 <= s1) old[j] = o2[s2];
        }
      }
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const int jj = 8 * h + j;
        const int s2 = s2_0 + jj;
        if (s2 >= 0 && s2 <= s1) {
          V2 v;
          v.x = val(re[jj]);
          v.y = val(im[jj]);
          if (add) {
            v.x += old[j].x;
            v.y += old[j].y;
          }
          o2[s2] = v;
        }
      }
    }
  }
}

// Undo the operand scales of float input: V(a, b0 + j) *= 2^(e_a + e_b).
template <int FMT>
__device__ __forceinline__ void scale_piece(uint32_t (&re)[32], uint32_t (&im)[32], const Params& p,
                                            int f, int a, int b0) {
  const unsigned* am = p.in_amax + static_cast<int64_t>(f) * p.n;
  const int ea = a < p.n ? scale_exp<FMT>(am[a]) : 0;
#pragma unroll
  for (int j = 0; j < 32; ++j) {
    const int b = b0 + j;
    const float sc = exp2i(ea + (b < p.n ? scale_exp<FMT>(am[b]) : 0));
    re[j] = __float_as_uint(__uint_as_float(re[j]) * sc);
    im[j] = __float_as_uint(__uint_as_float(im[j]) * sc);
  }
}

// FP64 block sums: acc64 = (first chunk and not accumulating ? 0 : acc64) +
// piece; the last chunk of the integration also stores its fp32 rounding.
__device__ __forceinline__ void store_piece_f64(const uint32_t (&re)[32], const uint32_t (&im)[32],
                                                const Params& p, int f, int a, int b0, bool first,
                                                bool last, uint64_t pol) {
  const int P = p.g.P;
  // Every lane of the warp joins the pairs path's exchanges; rows past n
  // (the ragged last block) only skip their memory accesses.
  const bool valid = a < p.n;
  if (!valid && !(P == 2 && p.pack == 1)) return;
  int s1 = a >> (P - 1), joff = 0, fr = f;
  const int p1 = a - s1 * P;
  if (p.pack > 1) {  // packed channels: real channel and stations
    const int j = s1 / p.Nr;
    joff = j * p.Nr;
    s1 -= joff;
    fr = f * p.pack + j;
  }
  const int64_t krow = static_cast<int64_t>(fr) * p.NBr + static_cast<int64_t>(s1) * (s1 + 1) / 2;
  const bool load_old = !first || p.accumulate;
  // The running sum outlives this drain unless it is the integration's last
  // one and calls do not accumulate.
  const bool keep = !last || p.accumulate;
  double2* ws = reinterpret_cast<double2*>(p.acc64);
  float2* out = static_cast<float2*>(p.out);
  if (P == 2 && p.pack == 1) {
    // As the int32 store's pairs path: the lanes of a station's two
    // polarisation rows (a, a ^ 1) exchange halves so that each holds one
    // whole baseline record {(0,0), (0,1), (1,0), (1,1)}: the p1 = 0 lane the
    // record of column station 2m, the p1 = 1 lane that of 2m + 1.  A lane
    // then moves 64 contiguous bytes of running sums (and 32 of output), and
    // a lane pair 128 contiguous bytes of one baseline row.
    const int s2_0 = b0 / 2;
    // Groups of MG records: the running sums of a group are loaded before
    // any of its stores (the compiler cannot move a load above a store to
    // the same buffer), so their memory latencies overlap.
    constexpr int MG = 2;
#pragma unroll
    for (int h = 0; h < 8 / MG; ++h) {
      double2 old[MG][4];
      if (load_old) {
#pragma unroll
        for (int mm = 0; mm < MG; ++mm) {
          const int s2 = s2_0 + 2 * (MG * h + mm) + p1;
          const bool ok = valid && s2 <= s1;
#pragma unroll
          for (int k = 0; k < 4; ++k)
            old[mm][k] = ok ? ws[(krow + s2) * 4 + k] : make_double2(0.0, 0.0);
        }
      }
#pragma unroll
      for (int mm = 0; mm < MG; ++mm) {
        const int m = MG * h + mm;
        float own[4], got[4];
#pragma unroll
        for (int q = 0; q < 2; ++q) {
          const float r0 = __uint_as_float(re[4 * m + q]), i0 = __uint_as_float(im[4 * m + q]);
          const float r1 = __uint_as_float(re[4 * m + 2 + q]), i1 = __uint_as_float(im[4 * m + 2 + q]);
          own[2 * q] = p1 ? r1 : r0;
          own[2 * q + 1] = p1 ? i1 : i0;
          got[2 * q] = __shfl_xor_sync(0xffffffffu, p1 ? r0 : r1, 1);
          got[2 * q + 1] = __shfl_xor_sync(0xffffffffu, p1 ? i0 : i1, 1);
        }
        // Products (p1', p2) of the record: row p1' = 0 from the p1 = 0 lane.
        double2 v[4];
#pragma unroll
        for (int q = 0; q < 2; ++q) {
          const float* r0 = p1 ? got : own;  // row 0 of the record
          const float* r1 = p1 ? own : got;  // row 1
          v[q] = make_double2(r0[2 * q], r0[2 * q + 1]);
          v[2 + q] = make_double2(r1[2 * q], r1[2 * q + 1]);
        }
        const int s2 = s2_0 + 2 * m + p1;
        if (!valid || s2 > s1) continue;
        double2* w4 = ws + (krow + s2) * 4;
        if (load_old) {
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            v[k].x += old[mm][k].x;
            v[k].y += old[mm][k].y;
          }
        }
        if (keep) {
#pragma unroll
          for (int k = 0; k < 4; ++k) w4[k] = v[k];
        }
        if (last) {
          uint32_t rec[8];
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            rec[2 * k] = __float_as_uint(static_cast<float>(v[k].x));
            rec[2 * k + 1] = __float_as_uint(static_cast<float>(v[k].y));
          }
          ptx::st_global_v8_hint(out + (krow + s2) * 4, rec, pol);
        }
      }
    }
    return;
  }
#pragma unroll
  for (int j = 0; j < 32; ++j) {
    const int b = b0 + j;
    const int s2v = b >> (P - 1), p2 = b - s2v * P, s2 = s2v - joff;
    if (s2 < 0 || s2 > s1) continue;
    const int64_t idx = (krow + s2) * P * P + p1 * P + p2;
    double2 v = make_double2(static_cast<double>(__uint_as_float(re[j])),
                             static_cast<double>(__uint_as_float(im[j])));
    if (load_old) {
      const double2 o = ws[idx];
      v.x += o.x;
      v.y += o.y;
    }
    if (!last || p.accumulate) ws[idx] = v;
    if (last) out[idx] = make_float2(static_cast<float>(v.x), static_cast<float>(v.y));
  }
}

// Transposed blocks (CTA pairs): this thread's row a lies in a row block
// above the piece's columns b0 .. b0 + 31 (every b > a), so the stored lower
// entries are the mirror ones, V[b][a] = conj(V[a][b]): baseline
// (s1, s2) = (s_b, s_a), polarisation product p_b * P + p_a.  Packed
// channels never occur here (they have one block row).
template <int WORD>
__device__ __forceinline__ void store_piece_tr(const uint32_t (&re)[32], const uint32_t (&im)[32],
                                               const Params& p, int f, int a, int b0, bool add,
                                               uint64_t pol) {
  constexpr bool IS_INT = WORD != kWordFloat;
  using T = typename std::conditional<IS_INT, int, float>::type;
  const Geometry& g = p.g;
  T* out = static_cast<T*>(p.out);
  const int P = g.P;
  const int sa = a >> (P - 1), pa = a - sa * P;
  // The stored word of the conjugate: int32 value or fp32 bits.
  auto re_bits = [](uint32_t u) -> uint32_t { return out_word<WORD>(u); };
  auto im_bits = [](uint32_t u) -> uint32_t {  // of -im
    if constexpr (IS_INT) {
      return 0u - out_word<WORD>(u);
    } else {
      return u ^ 0x80000000u;
    }
  };
  const bool pairs = P == 2 && !add && (reinterpret_cast<uintptr_t>(out) & 31) == 0;
  if (pairs) {
    // Lanes (2i, 2i + 1) hold pols 0 and 1 of station s_a.  For column
    // stations s_b0 + 2k (written by the pa = 0 lane) and s_b0 + 2k + 1 (by
    // the pa = 1 lane) each lane needs its partner's two products of that
    // column station: one exchange of 4 words per k gives both lanes whole
    // 32-byte records, {(0,0), (0,1), (1,0), (1,1)} x {re, im}.
    const bool row_ok = a < p.n;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      uint32_t own[4], got[4];
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        // Columns 4k + q (station 2k) and 4k + 2 + q (station 2k + 1): the
        // pa = 0 lane keeps the first and sends the second, pa = 1 the reverse.
        const uint32_t r0 = re_bits(re[4 * k + q]), i0 = im_bits(im[4 * k + q]);
        const uint32_t r1 = re_bits(re[4 * k + 2 + q]), i1 = im_bits(im[4 * k + 2 + q]);
        own[2 * q] = pa ? r1 : r0;
        own[2 * q + 1] = pa ? i1 : i0;
        got[2 * q] = __shfl_xor_sync(0xffffffffu, pa ? r0 : r1, 1);
        got[2 * q + 1] = __shfl_xor_sync(0xffffffffu, pa ? i0 : i1, 1);
      }
      uint32_t rec[8];
#pragma unroll
      for (int q = 0; q < 2; ++q) {  // products (p_b = q, p_a = 0) and (q, 1)
        rec[4 * q + 0] = pa ? got[2 * q] : own[2 * q];
        rec[4 * q + 1] = pa ? got[2 * q + 1] : own[2 * q + 1];
        rec[4 * q + 2] = pa ? own[2 * q] : got[2 * q];
        rec[4 * q + 3] = pa ? own[2 * q + 1] : got[2 * q + 1];
      }
      const int sb = b0 / 2 + 2 * k + pa;
      if (row_ok && sb < g.N) {
        const int64_t rec_idx =
            static_cast<int64_t>(f) * p.NBr + static_cast<int64_t>(sb) * (sb + 1) / 2 + sa;
        ptx::st_global_v8_hint(reinterpret_cast<uint32_t*>(out) + rec_idx * 8, rec, pol);
      }
    }
    return;
  }
  if (a >= p.n) return;
#pragma unroll
  for (int j = 0; j < 32; ++j) {
    const int b = b0 + j;
    if (b >= p.n) continue;
    const int sb = b >> (P - 1), pb = b - sb * P;
    const int64_t idx =
        ((static_cast<int64_t>(f) * p.NBr + static_cast<int64_t>(sb) * (sb + 1) / 2 + sa) * P + pb) * P + pa;
    uint32_t w[2] = {re_bits(re[j]), im_bits(im[j])};
    T* o = out + idx * 2;
    if (add) {
      o[0] += *reinterpret_cast<const T*>(&w[0]);
      o[1] += *reinterpret_cast<const T*>(&w[1]);
    } else if constexpr (IS_INT) {
      *reinterpret_cast<int2*>(o) = make_int2(static_cast<int>(w[0]), static_cast<int>(w[1]));
    } else {
      *reinterpret_cast<float2*>(o) = make_float2(__uint_as_float(w[0]), __uint_as_float(w[1]));
    }
  }
}

// FP64 block sums of a transposed block (see store_piece_f64, store_piece_tr).
__device__ __forceinline__ void store_piece_f64_tr(const uint32_t (&re)[32], const uint32_t (&im)[32],
                                                   const Params& p, int f, int a, int b0, bool first,
                                                   bool last) {
  if (a >= p.n) return;
  const int P = p.g.P;
  const int sa = a >> (P - 1), pa = a - sa * P;
  const bool load_old = !first || p.accumulate;
  double2* ws = reinterpret_cast<double2*>(p.acc64);
  float2* out = static_cast<float2*>(p.out);
#pragma unroll
  for (int j = 0; j < 32; ++j) {
    const int b = b0 + j;
    if (b >= p.n) continue;
    const int sb = b >> (P - 1), pb = b - sb * P;
    const int64_t idx =
        ((static_cast<int64_t>(f) * p.NBr + static_cast<int64_t>(sb) * (sb + 1) / 2 + sa) * P + pb) * P + pa;
    double2 v = make_double2(static_cast<double>(__uint_as_float(re[j])),
                             -static_cast<double>(__uint_as_float(im[j])));
    if (load_old) {
      const double2 o = ws[idx];
      v.x += o.x;
      v.y += o.y;
    }
    if (!last || p.accumulate) ws[idx] = v;
    if (last) out[idx] = make_float2(static_cast<float>(v.x), static_cast<float>(v.y));
  }
}

// ------------------------------------------------------------------ kernel

// stage_acc flags: the step opens an accumulation group (closing the one that
// is open), or is the last step of its group.
// A diagonal step has one operand pair (kAccSame).  The MMA's N sits above.
enum : int { kAccStart = 1, kAccEnd = 2, kAccSame = 4, kAccNShift = 8 };

// Per-launch constants of the item loop: CTA pairs walk the items by
// cluster, single CTAs by block.
template <int SHAPE>
__device__ __forceinline__ long long item_first() {
  return SHAPE == kShapePair ? static_cast<long long>(blockIdx.x >> 1) : static_cast<long long>(blockIdx.x);
}
template <int SHAPE>
__device__ __forceinline__ long long item_stride() {
  return SHAPE == kShapePair ? static_cast<long long>(gridDim.x >> 1) : static_cast<long long>(gridDim.x);
}

template <bool IS_INT, int DT, int FMT, bool MULTI, int SHAPE, int IN>
__device__ __forceinline__ void planar_body(const Batch& bt) {
  constexpr bool PAIR = SHAPE == kShapePair;
  constexpr bool WIDE = SHAPE == kShapeWide;
  using C = Cfg<SHAPE, FMT, DT>;
  constexpr int kStages = C::kStages;
  constexpr int kSteps = FmtT<FMT, SHAPE>::kSteps;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                             ~static_cast<uintptr_t>(1023));
  const uint32_t sbase = ptx::smem_u32(smem);
  const uint32_t bar0 = sbase + C::kBarOff;
  auto full_bar = [&](int s) { return bar0 + 8u * s; };
  auto empty_bar = [&](int s) { return bar0 + 8u * (kStages + s); };
  auto pfull_bar = [&](int s) { return bar0 + 8u * (2 * kStages + s); };  // PAIR only
  constexpr int kB = (PAIR ? 3 : 2) * kStages;
  auto accf_bar = [&](int b) { return bar0 + 8u * (kB + b); };
  auto acce_bar = [&](int b) { return bar0 + 8u * (kB + 2 + b); };
  const uint32_t drain_bar = bar0 + 8u * (kB + 4);
  auto conv_bar = [&](int w) { return bar0 + 8u * (kB + 5 + w); };
  uint32_t* tmem_holder = reinterpret_cast<uint32_t*>(smem + C::kBarOff + C::kNumBars * 8);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_holder + 1);
  // What stage s's step does to the accumulation (kAccStart, kAccEnd): the
  // producer (which has waited for the step's segment) writes it before the
  // stage's arrive, so the MMA thread reads it after its wait with no global
  // round trip of its own.
  volatile int* stage_acc = reinterpret_cast<volatile int*>(tmem_holder + 2);
  // 8-bit input: is the group in accumulator set b the last one of its item?
  // The MMA warp, which learns from the stages where groups end, writes it
  // before it arrives on accf (the second arrival beside the MMAs' own); the
  // epilogue reads it before it releases the set.
  uint32_t* acc_last = tmem_holder + 2 + kStages;

  const int warp = __shfl_sync(0xffffffffu, static_cast<int>(threadIdx.x >> 5), 0);  // (known uniform)
  const int lane = threadIdx.x & 31;
  const uint32_t rank = PAIR ? ptx::cluster_ctarank() : 0u;
  const bool leader = rank == 0;

  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) {
      ptx::mbar_init(full_bar(s), 1);
      ptx::mbar_init(empty_bar(s), 1);
      if (PAIR) ptx::mbar_init(pfull_bar(s), 1);
    }
    for (int b = 0; b < 2; ++b) {
      ptx::mbar_init(accf_bar(b), IS_INT ? 2 : 1);
      ptx::mbar_init(acce_bar(b), (PAIR ? 2 : 1) * kNumEpiWarps);
    }
    ptx::mbar_init(drain_bar, 1);
    for (int w = 0; w < conv_warps<FMT, DT>(); ++w) ptx::mbar_init(conv_bar(w), 1);
    *abort_flag = 0;
    ptx::fence_mbar_init();
    ptx::fence_proxy_async_smem();
  }
  if (warp == 1) {
    if constexpr (PAIR) {
      ptx::tmem_alloc_pair(ptx::smem_u32(tmem_holder), kTmemCols);
      ptx::tmem_relinquish_pair();
    } else {
      ptx::tmem_alloc(ptx::smem_u32(tmem_holder), kTmemCols);
      ptx::tmem_relinquish();
    }
  }
  ptx::tc_fence_before();
  __syncthreads();
  if constexpr (PAIR) ptx::cluster_sync();  // both CTAs' barriers exist before any remote arrive
  ptx::tc_fence_after();
  const uint32_t tmem = *tmem_holder;

  // Hi/lo operands: 22-bit products lose accuracy in a long fp32 TMEM
  // accumulation, so the MMA restarts its accumulator (buffer 0) every
  // 64-sample K-block and the epilogue adds each block into a round-to-nearest
  // fp32 running sum held in TMEM columns 256..511 (not with 128 x 256 items,
  // whose accumulators fill the 512 columns).
  constexpr bool kTmemSum = FMT == kFmtHiLo;
  static_assert(!(kTmemSum && WIDE), "hi/lo operands need TMEM columns 256..511 for their sums");
  // One accumulator set in TMEM (no double buffer) for 128 x 256 items:
  // D_re in columns 0..255, D_im in 256..511.  Other shapes alternate two
  // sets {D_re, D_im} of 128 + 128 columns.
  constexpr uint32_t kImCol = WIDE ? 256 : 128;  // of D_im (D_re is at column 0 of its set)
  constexpr bool kOneSet = kTmemSum || WIDE;
  constexpr int TB = FmtT<FMT, SHAPE>::kTile;
  const ptx::WaitCtl wc{bt.sub[0].timeout_ns, bt.sub[0].status, abort_flag};
  const long long nitems = table_end<MULTI>(bt.item_base, bt.nsub);
  const long long it0 = item_first<SHAPE>(), istep = item_stride<SHAPE>();

  if (warp == 0) {
    // ------------------------------------------------------------ producer
    // The whole warp walks the items; lane 0 waits for stages, releases
    // segments and issues the copies, and the lanes together look at up to 32
    // segments of a channel at a time (one round trip to L2 for all of them).
    int stage = 0;
    uint32_t phase = 0;
    long long issued = 0;  // stages filled so far
    // Parity of the phase that stage s's last fill (of any so far) runs in.
    auto fill_phase = [&](int s) { return s < stage ? phase : phase ^ 1u; };
    // Lane 0.  Bit s: stage s holds this item's last step of a segment, whose
    // done counter rel[s] is released once the stage's MMAs have completed.
    uint32_t rel_mask = 0;
    unsigned* rel[kStages];
    auto release = [&](int s) {
      red_release_add(rel[s], 1u);
      rel_mask &= ~(1u << s);
    };
    bool ok = true;
    int ready_chan = -1, ready_sb = -1;
    const uint64_t pol_last = ptx::l2_policy_evict_last();  // tiles are shared by the channel's blocks
    for (Item x = item_start<MULTI>(bt, it0, nitems); ok && x.it < nitems;
         item_step<MULTI>(bt, x, istep, nitems)) {
      const Params& p = bt.sub[x.sb];
      const Blk k = item_block<SHAPE>(p, x, rank);
      int width;
      const int G0 = seg_first(p, k.f, &width);
      int slot = G0 - fast_div(G0, p.ring_slots, p.mag_slots) * p.ring_slots;
      const bool new_chan = k.f != ready_chan || x.sb != ready_sb;
      ready_chan = k.f;
      ready_sb = x.sb;
      const bool diag = SHAPE == kShape128 && k.a == k.b;
      // MMA shape.  128 x 128: M = 128 rows, N trimmed to the block's valid
      // columns (rounded up to 16), so ragged edge blocks skip the zero
      // columns.  Pairs: M = 256 (both row blocks), N = 128, 64 per CTA.
      // 128 x 256: N = 128 + the second block's valid columns (it sits right
      // after the first in shared memory, whatever their block indices).
      const bool two = WIDE && k.b2 >= 0;
      const int mma_n = PAIR ? kBlk : (((two ? kBlk : 0) + min(kBlk, p.n - (two ? k.b2 : k.b) * kBlk) + 15) & ~15);
      const int64_t kt_step = static_cast<int64_t>(p.nib) * FmtT<FMT, SHAPE>::kKbBytes;  // between K-tiles
      const int64_t slot_step = p.nkt * kt_step;
      const int64_t a_off = static_cast<int64_t>(k.a) * FmtT<FMT, SHAPE>::kKbBytes;
      const int64_t b_off = static_cast<int64_t>(k.b) * FmtT<FMT, SHAPE>::kKbBytes;
      const uint8_t* slot_base = p.ring + slot * slot_step;
      unsigned grow = 0, sum = 0;  // 8-bit input: exact-chunk bookkeeping
      int f_left = 0;              // float input: K-blocks left in the fp32 chunk
      int seg = 0, kl = 0;         // segment, K-block in it
      // The window of 32 segments that seg is in: which are known to be
      // converted, and (lane l: the window's segment l) their growth.
      uint32_t known = 0;
      unsigned my_grow = 0;
      // Segments of the window from seg on.
      auto look = [&]() {
        const int s = (seg & ~31) + lane;
        bool r = s >= seg && s < p.nseg;
        if (r && new_chan) {
          const int G = G0 + s * width, gen = fast_div(G, p.ring_slots, p.mag_slots);
          r = ld_acquire(p.ready + G - gen * p.ring_slots) >=
              static_cast<unsigned>(gen + 1) * static_cast<unsigned>(p.seg_units);
        }
        // (A converted segment's max |x| is final.)
        if (IS_INT && r) my_grow = kblock_growth(p, G0 + s * width);
        known |= __ballot_sync(0xffffffffu, r);
        __syncwarp();  // what lane l acquired is ordered before lane 0's copies
      };
      for (int kb = 0; ok && kb < p.nkb; ++kb) {
        if (kl == 0) {
          // A new segment: wait until it is converted.
          if ((seg & 31) == 0) {
            known = 0;
            look();
          }
          const uint64_t t0 = (known >> (seg & 31) & 1u) ? 0 : ptx::globaltimer();
          while (!(known >> (seg & 31) & 1u)) {
            // Meanwhile, release what has completed.
            if (lane == 0)
              for (int s = 0; s < kStages; ++s)
                if ((rel_mask >> s & 1u) && ptx::mbar_test_wait(empty_bar(s), fill_phase(s))) release(s);
            __nanosleep(32);
            look();
            const bool over = !(known >> (seg & 31) & 1u) && lane == 0 && wait_given_up(p, t0, abort_flag);
            if (__any_sync(0xffffffffu, over)) {
              ok = false;
              break;
            }
          }
          if (!ok) break;
          if constexpr (IS_INT) grow = __shfl_sync(0xffffffffu, my_grow, seg & 31);
        }
        int acc = kb == 0 ? kAccStart : 0;
        if constexpr (IS_INT) {
          if (kb > 0 && sum + grow > kExactSum) {
            acc = kAccStart;
            sum = 0;
          }
          sum += grow;
        } else {
          if (f_left == 0) {
            acc = kAccStart;
            f_left = p.f_chunk_kb;
          }
          --f_left;
          if (kTmemSum) acc = kAccStart;
        }
        const bool acc_end = kb + 1 == p.nkb || (!IS_INT && (kTmemSum || f_left == 0));
        const bool seg_end = kl + 1 == p.seg_kb || kb + 1 == p.nkb;
        for (int st = 0; ok && st < kSteps; ++st) {
          // HI/LO operand pairs j = 0, 1, 2 of a K-block: (H, H), (L, H), (H, L).
          constexpr int kSpj = FmtT<FMT, SHAPE>::kSplit;
          const int j = st / kSpj, half = st % kSpj;
          const uint8_t* ar = slot_base + (kl + (j == 1 ? p.seg_kb : 0)) * kt_step + a_off + half * 2 * TB;
          const uint8_t* br = slot_base + (kl + (j == 2 ? p.seg_kb : 0)) * kt_step + b_off + half * 2 * TB;
          const bool jlast = st + 1 == kSteps;
          const bool same = diag && (FMT != kFmtHiLo || j == 0);
          const int word = (st == 0 ? acc : 0) | (jlast && acc_end ? kAccEnd : 0) | (same ? kAccSame : 0) |
                           mma_n << kAccNShift;
          const uint32_t dst = sbase + stage * C::kStageBytes;
          const uint32_t fb = full_bar(stage);
          bool got = true;
          if (lane == 0) {
            got = ptx::wait_bounded(empty_bar(stage), phase ^ 1u, wc);
            if (got) {
              // The MMAs of an item's last step of a segment have read it.
              if (rel_mask >> stage & 1u) release(stage);
              stage_acc[stage] = word;  // published by the arrive below
              if (jlast && seg_end && leader) {
                rel[stage] = p.done + slot;
                rel_mask |= 1u << stage;
              }
              if constexpr (PAIR) {
                // A: this CTA's row block (not needed by an idle CTA); B: this
                // CTA's half of the column block (always: the leader's MMA reads it).
                constexpr int HB = TB / 2;
                ptx::mbar_arrive_expect_tx(fb, (k.idle ? 1 : 3) * TB);
                if (!k.idle) ptx::bulk_load_hint(dst, ar, 2 * TB, fb, pol_last);
                ptx::bulk_load_hint(dst + 2 * TB, br + rank * HB, HB, fb, pol_last);
                ptx::bulk_load_hint(dst + 2 * TB + HB, br + TB + rank * HB, HB, fb, pol_last);
              } else if constexpr (WIDE) {
                // Ar, Ai; then Br of both column blocks back to back (one 256-row
                // operand: the second tile starts 16 groups on), and Bi likewise.
                ptx::mbar_arrive_expect_tx(fb, two ? 6 * TB : 4 * TB);
                ptx::bulk_load_hint(dst, ar, 2 * TB, fb, pol_last);
                ptx::bulk_load_hint(dst + 2 * TB, br, TB, fb, pol_last);
                ptx::bulk_load_hint(dst + 4 * TB, br + TB, TB, fb, pol_last);
                if (two) {
                  const uint8_t* br2 = br + static_cast<int64_t>(k.b2 - k.b) * FmtT<FMT, SHAPE>::kKbBytes;
                  ptx::bulk_load_hint(dst + 3 * TB, br2, TB, fb, pol_last);
                  ptx::bulk_load_hint(dst + 5 * TB, br2 + TB, TB, fb, pol_last);
                }
              } else {
                constexpr int OB = 2 * TB;  // one operand
                ptx::mbar_arrive_expect_tx(fb, same ? OB : 2 * OB);
                ptx::bulk_load_hint(dst, ar, OB, fb, pol_last);
                if (!same) ptx::bulk_load_hint(dst + OB, br, OB, fb, pol_last);
              }
            }
          }
          if (!__all_sync(0xffffffffu, got)) {
            ok = false;
            break;
          }
          ++issued;
          if (++stage == kStages) {
            stage = 0;
            phase ^= 1u;
          }
        }
        if (++kl == p.seg_kb) {
          kl = 0;
          ++seg;
          slot += width;
          while (slot >= p.ring_slots) slot -= p.ring_slots;
          slot_base = p.ring + slot * slot_step;
        }
      }
    }
    if (lane == 0) {
      // The last segments' releases: other CTAs' converters may wait for them.
      for (int s = 0; ok && s < kStages; ++s) {
        if (!(rel_mask >> s & 1u)) continue;
        if (ptx::wait_bounded(empty_bar(s), fill_phase(s), wc))
          release(s);
        else
          ok = false;
      }
      if (!ok) {
        for (int s = 0; s < kStages; ++s) {
          if (issued <= s) continue;
          const uint64_t t0 = ptx::globaltimer();
          while (!ptx::mbar_try_wait(full_bar(s), fill_phase(s)) &&
                 ptx::globaltimer() - t0 < wc.timeout_ns) {
          }
        }
      }
    }
    __syncwarp();
  } else if (warp == 1 && PAIR && !leader) {
    // ------------------------------------------------ peer relay (pairs)
    // Forwards each completed stage of this CTA to the leader's pfull.
    if (lane == 0) {
      int stage = 0;
      uint32_t phase = 0;
      bool ok = true;
      int sb = 0;
      for (long long it = it0; ok && it < nitems; it += istep) {
        sb = advance_sub<MULTI>(bt.item_base, bt.nsub, it, sb);
        const Params& p = bt.sub[sb];
        for (int st = 0; st < p.nkb * kSteps; ++st) {
          if (!ptx::wait_bounded(full_bar(stage), phase, wc)) {
            ok = false;
            break;
          }
          ptx::mbar_arrive_remote(ptx::mapa_shared(pfull_bar(stage), 0));
          if (++stage == kStages) {
            stage = 0;
            phase ^= 1u;
          }
        }
      }
    }
  } else if (warp == 1) {
    // ---------------------------------------------------------- MMA issuer
    // The whole warp walks the stages, so that loop state and descriptors are
    // warp-uniform (uniform registers, which tcgen05.mma takes them from); one
    // elected lane issues.  What the thread does between the last MMA of a
    // stage and the first of the next is not hidden by the MMA queue: a stage
    // cost about 600 cycles more than its MMAs when one lane ran this loop and
    // worked out each item's coordinates itself.
    const bool issuer = ptx::elect_one();
    int stage = 0;
    uint32_t phase = 0;
    uint32_t u = 0;
    bool ok = true;
    int sb = 0;
    // Accumulation groups: an exact chunk (8-bit input), an fp32 chunk, or one
    // K-block when the epilogue sums 64-sample fp32 blocks in TMEM (buffer 0
    // only).  The producer says where they start and, where it knows (not for
    // 8-bit chunks, whose end depends on the next segment's values), end.
    auto commit_acc = [&](uint32_t ab, bool last) {
      if (issuer) {
        if constexpr (IS_INT) {
          *reinterpret_cast<volatile uint32_t*>(acc_last + ab) = last ? 1u : 0u;
          ptx::mbar_arrive(accf_bar(ab));
          if constexpr (PAIR) {
            ptx::st_shared_remote(ptx::mapa_shared(ptx::smem_u32(acc_last + ab), 1), last ? 1u : 0u);
            ptx::mbar_arrive_remote(ptx::mapa_shared(accf_bar(ab), 1));
          }
        }
        if constexpr (PAIR) {
          ptx::mma_commit_pair_mc(accf_bar(ab), 0x3);
        } else {
          ptx::mma_commit(accf_bar(ab));
        }
      }
    };
    // Descriptors of stage 0's Ar; the other operands and stages and the
    // K-steps add their byte offsets (16-byte units) to the address field,
    // which cannot carry: every shared-memory address is below 256 KiB.
    const uint64_t desc0 = ptx::interleave_kmajor_desc(sbase, kCoreBytes, FmtT<FMT, SHAPE>::kSbo);
    constexpr uint64_t kStageDesc = C::kStageBytes >> 4, kTileDesc = TB >> 4;
    // The next stage's word, once it is known to be full: looked up while the
    // MMA queue still holds work, so that little but the issue itself lies
    // between two stages' MMAs.
    bool ahead = false;
    uint32_t word = 0;
    for (long long it = it0; ok && it < nitems; it += istep) {
      sb = advance_sub<MULTI>(bt.item_base, bt.nsub, it, sb);
      const int nsteps = bt.sub[sb].nkb * kSteps;
      bool open = false;
      uint32_t ab = 0, d_acc = 0, started = 0;
      for (int st = 0; st < nsteps; ++st) {
        if (!ahead) {
          const bool got = ptx::wait_bounded(full_bar(stage), phase, wc) &&
                           (!PAIR || ptx::wait_bounded(pfull_bar(stage), phase, wc));
          if (!__all_sync(0xffffffffu, got)) {
            ok = false;
            break;
          }
          word = __shfl_sync(0xffffffffu, static_cast<uint32_t>(stage_acc[stage]), 0);
        }
        if (word & kAccStart) {
          if (open) {
            commit_acc(ab, false);
            ++u;
          }
          ab = kOneSet ? 0u : (u & 1u);
          const uint32_t ap = kOneSet ? (u & 1u) : ((u >> 1) & 1u);
          const bool drained = ptx::wait_bounded(acce_bar(ab), ap ^ 1u, wc);
          if (!__all_sync(0xffffffffu, drained)) {
            ok = false;
            break;
          }
          d_acc = tmem + ab * 256;
          open = true;
          started = 0;
        }
        ptx::tc_fence_after();
        const uint32_t d_re = d_acc, d_im = d_acc + kImCol;
        const int mma_n = static_cast<int>(word >> kAccNShift);
        const uint32_t idesc = ptx::idesc_f16_f32(PAIR ? 2 * kBlk : kBlk, mma_n);
        const uint32_t idesc_negb = idesc | (1u << 14);
        const uint64_t dar0 = desc0 + static_cast<uint64_t>(stage) * kStageDesc;
        const bool same = !PAIR && !WIDE && (word & kAccSame);
        const uint64_t dbr0 = same ? dar0 : dar0 + 2 * kTileDesc;
        // Four MMAs per K-step, and every MMA into an accumulator has the same
        // shape, as every step of an item has: only then does PTX order
        // back-to-back MMAs on it.  (One 128 x 256 MMA for Im += Ai Br^T and
        // Re += Ai Bi^T beside two of 128 x 128 would read 28 instead of 32 KiB
        // of shared memory per K-step, 1025 cycles per 64 samples against 1114
        // alone, but mixes shapes on both accumulators.  In the whole kernel it
        // gave nothing: 256 stations, F=1024, T=1000 1.00 ms either way.)
        // K-step kk: 16-byte chunks 2kk and 2kk + 1 (16 fp16 or 32 e4m3 samples).
        auto kstep = [&](int kk) {
          const uint32_t acc = kk > 0 ? 1u : started;
          const uint64_t kd = static_cast<uint64_t>(kk * 2 * kCoreBytes) >> 4;
          const uint64_t dar = dar0 + kd, dai = dar + kTileDesc;
          const uint64_t dbr = dbr0 + kd;
          const uint64_t dbi = dbr + (PAIR ? kTileDesc / 2 : (WIDE ? 2 : 1) * kTileDesc);
          if constexpr (PAIR && FMT == kFmtF8) {
            ptx::mma_f8_ss_pair(d_re, dar, dbr, idesc, acc);       // Re += Ar Br^T
            ptx::mma_f8_ss_pair(d_re, dai, dbi, idesc, 1u);        // Re += Ai Bi^T
            ptx::mma_f8_ss_pair(d_im, dai, dbr, idesc, acc);       // Im += Ai Br^T
            ptx::mma_f8_ss_pair(d_im, dar, dbi, idesc_negb, 1u);   // Im -= Ar Bi^T
          } else if constexpr (PAIR) {
            ptx::mma_f16_ss_pair(d_re, dar, dbr, idesc, acc);
            ptx::mma_f16_ss_pair(d_re, dai, dbi, idesc, 1u);
            ptx::mma_f16_ss_pair(d_im, dai, dbr, idesc, acc);
            ptx::mma_f16_ss_pair(d_im, dar, dbi, idesc_negb, 1u);
          } else if constexpr (FMT == kFmtF8) {
            ptx::mma_f8_ss(d_re, dar, dbr, idesc, acc);
            ptx::mma_f8_ss(d_re, dai, dbi, idesc, 1u);
            ptx::mma_f8_ss(d_im, dai, dbr, idesc, acc);
            ptx::mma_f8_ss(d_im, dar, dbi, idesc_negb, 1u);
          } else {
            ptx::mma_f16_ss(d_re, dar, dbr, idesc, acc);
            ptx::mma_f16_ss(d_re, dai, dbi, idesc, 1u);
            ptx::mma_f16_ss(d_im, dai, dbr, idesc, acc);
            ptx::mma_f16_ss(d_im, dar, dbi, idesc_negb, 1u);
          }
        };
        constexpr int kAll = FmtT<FMT, SHAPE>::kChunks / 2;
        if (issuer) {
#pragma unroll
          for (int kk = 0; kk < kAll - 1; ++kk) kstep(kk);
        }
        __syncwarp();
        const int nstage = stage + 1 == kStages ? 0 : stage + 1;
        const uint32_t nphase = stage + 1 == kStages ? phase ^ 1u : phase;
        ahead = ptx::mbar_test_wait(full_bar(nstage), nphase) &&
                (!PAIR || ptx::mbar_test_wait(pfull_bar(nstage), nphase));
        ahead = __all_sync(0xffffffffu, ahead);
        uint32_t next_word = 0;
        if (ahead) next_word = __shfl_sync(0xffffffffu, static_cast<uint32_t>(stage_acc[nstage]), 0);
        if (issuer) {
          kstep(kAll - 1);
          if constexpr (PAIR) {
            ptx::mma_commit_pair_mc(empty_bar(stage), 0x3);
          } else {
            ptx::mma_commit(empty_bar(stage));
          }
        }
        started = 1;
        if (word & kAccEnd) {  // (8-bit input: of the item's last group only)
          commit_acc(ab, true);
          ++u;
          open = false;
        }
        word = next_word;
        stage = nstage;
        phase = nphase;
      }
    }
    if (!ok && issuer) {
      // The MMAs issued so far complete before TMEM is freed (bounded).
      if constexpr (PAIR) {
        ptx::mma_commit_pair_mc(drain_bar, 0x1);
      } else {
        ptx::mma_commit(drain_bar);
      }
      const uint64_t t0 = ptx::globaltimer();
      while (!ptx::mbar_try_wait(drain_bar, 0) && ptx::globaltimer() - t0 < wc.timeout_ns) {
      }
    }
    __syncwarp();
  } else if (warp < 2 + kNumEpiWarps) {
    // ------------------------------------------------------------ epilogue
    const int q = warp & 3;
    const uint32_t t_lanes = tmem + (static_cast<uint32_t>(q * 32) << 16);
    uint32_t u = 0;
    bool ok = true;
    // The visibilities are written once: first in line for L2 replacement.
    const uint64_t pol_out = ptx::l2_policy_evict_first();
    // Accumulator b has been read: local arrive, or remote on the leader's barrier.
    auto release_acc = [&](uint32_t ab) {
      ptx::tc_fence_before();
      __syncwarp();
      if (lane == 0) {
        if (!PAIR || leader)
          ptx::mbar_arrive(acce_bar(ab));
        else
          ptx::mbar_arrive_remote(ptx::mapa_shared(acce_bar(ab), 0));
      }
    };
    for (Item x = item_start<MULTI>(bt, it0, nitems); ok && x.it < nitems;
         item_step<MULTI>(bt, x, istep, nitems)) {
      const Params& p = bt.sub[x.sb];
      const int P = p.g.P;
      const Blk k = item_block<SHAPE>(p, x, rank);
      const int f = k.f;
      const int a = k.a * kBlk + q * 32 + lane;  // this thread's row input
      // The item's column blocks and, per block, the pieces piece0..last this
      // warp stores: for a block on or below the diagonal those that can reach
      // the lower station triangle (packed channels: only from the first
      // column of the lowest row's real channel on); for a mirrored block
      // every piece with a valid column.
      const int nblk = (WIDE && k.b2 >= 0) ? 2 : 1;
      int cb[2] = {k.b, k.b2}, first_p[2] = {0, 0}, last_p[2] = {-1, -1};
      for (int j = 0; j < nblk; ++j) {
        const int b = cb[j];
        if (k.idle) continue;
        if (b > k.a) {
          last_p[j] = min(kBlk / 32 - 1, (p.n - 1 - b * kBlk) >> 5);
        } else {
          // The last input of this warp's highest station row.
          const int hi = min(p.n - 1, k.a * kBlk + q * 32 + 31);
          last_p[j] = max(-1, min(kBlk / 32 - 1, (hi - b * kBlk) >> 5));
          if (p.pack > 1) {
            const int col0 = (k.a * kBlk + q * 32) / P / p.Nr * p.Nr * P;  // first column of that channel
            first_p[j] = max(0, (col0 - b * kBlk) / 32);
            if (first_p[j] > last_p[j]) last_p[j] = -1;  // no row of this warp is valid
          }
        }
      }
      // The last block with pieces to read releases the accumulator after them.
      const int jlast = (nblk == 2 && last_p[1] >= 0) ? 1 : (last_p[0] >= 0 ? 0 : -1);
      // The item's chunks: of f_chunk_kb K-blocks (float input), or until the
      // MMA warp says that an accumulator holds the last one (8-bit input, one
      // group each).
      int kb0 = 0;
      bool last_chunk = false;
      for (int ch = 0; ok && !last_chunk; ++ch) {
        const int kb1 = IS_INT ? kb0 + 1 : min(p.nkb, kb0 + p.f_chunk_kb);
        if (!IS_INT) last_chunk = kb1 == p.nkb;
        const int gstep = kTmemSum ? 1 : (kb1 - kb0);
        const bool add = p.accumulate || ch > 0;
        // FP64 block sums: chunks pair off, (0, 1), (2, 3), ...  The first
        // chunk of a pair stays in its TMEM accumulator (`hold`); the second's
        // drain adds it in fp32 (a correctly rounded sum of the two partials,
        // what an fp64 add rounded back would give) and updates the float64
        // running sum once per pair: half the passes over it, none at all for
        // an integration of two chunks.  Needs the two accumulator sets.
        const bool f64pair = !IS_INT && !kOneSet && p.acc64 != nullptr;
        const bool hold = f64pair && (ch % 2 == 0) && !last_chunk;
        const bool paired = f64pair && (ch % 2 == 1);
        const bool first = f64pair ? ch < 2 : ch == 0;
        for (int g0 = kb0; g0 < kb1; g0 += gstep) {
          // TMEM running sum: the first group of a chunk starts it, the last
          // one is stored; groups in between only add into it.
          const bool gfirst = g0 == kb0, glast = g0 + gstep >= kb1;
          const uint32_t ab = kOneSet ? 0u : (u & 1u);
          const uint32_t ap = kOneSet ? (u & 1u) : ((u >> 1) & 1u);
          if constexpr (!IS_INT) {
            // FP64 block sums: while the MMAs run, bring into L2 the running
            // sums this drain will read: each lane of a row's pair prefetches
            // half of the row's records in the block (one bulk request).
            if (p.acc64 && !hold && (!first || p.accumulate) && glast && P == 2 && p.pack == 1 && a < p.n) {
              const int s1 = a / 2;
              const int64_t krow = static_cast<int64_t>(f) * p.NBr + static_cast<int64_t>(s1) * (s1 + 1) / 2;
              for (int j = 0; j < nblk; ++j) {
                const int b = cb[j];
                if (b > k.a) continue;  // mirrored blocks write other rows
                const int lo = b * (kBlk / 2), hi = min(b * (kBlk / 2) + kBlk / 2 - 1, s1);
                const int half = (hi - lo + 2) / 2;
                const int from = lo + (a & 1) * half, cnt = min(half, hi - from + 1);
                if (cnt > 0)
                  ptx::bulk_prefetch_l2(reinterpret_cast<const double2*>(p.acc64) + (krow + from) * 4,
                                        static_cast<uint32_t>(cnt) * 64u);
              }
            }
          }
          const bool got = ptx::wait_bounded(accf_bar(ab), ap, wc);
          if (!__all_sync(0xffffffffu, got)) {
            ok = false;
            break;
          }
          if constexpr (IS_INT) {
            if (PAIR) ptx::mbar_acquire_cluster(accf_bar(ab), ap);  // (the peer's word comes from the leader)
            last_chunk = *reinterpret_cast<volatile uint32_t*>(acc_last + ab) != 0;
          }
          ptx::tc_fence_after();
          if (hold) {  // drained with the next chunk
            ++u;
            continue;
          }
          if (paired) {
            // Add the held chunk into this one inside TMEM and free it at
            // once, so the next item's MMAs need not wait for the stores.
            for (int j = 0; j < nblk; ++j) {
              const uint32_t c_re = ab * 256, c_im = ab * 256 + kImCol;
              const uint32_t h_re = (ab ^ 1u) * 256, h_im = (ab ^ 1u) * 256 + kImCol;
#pragma unroll 1
              for (int piece = first_p[j]; piece <= last_p[j]; ++piece) {
                uint32_t vr[32], vi[32], sr[32], si[32];
                ptx::tmem_ld_32x32b_x32(t_lanes + c_re + piece * 32, vr);
                ptx::tmem_ld_32x32b_x32(t_lanes + c_im + piece * 32, vi);
                ptx::tmem_ld_32x32b_x32(t_lanes + h_re + piece * 32, sr);
                ptx::tmem_ld_32x32b_x32(t_lanes + h_im + piece * 32, si);
                ptx::tmem_wait_ld();
#pragma unroll
                for (int jj = 0; jj < 32; ++jj) {
                  vr[jj] = __float_as_uint(__uint_as_float(vr[jj]) + __uint_as_float(sr[jj]));
                  vi[jj] = __float_as_uint(__uint_as_float(vi[jj]) + __uint_as_float(si[jj]));
                }
                ptx::tmem_st_32x32b_x32(t_lanes + c_re + piece * 32, vr);
                ptx::tmem_st_32x32b_x32(t_lanes + c_im + piece * 32, vi);
              }
            }
            ptx::tmem_wait_st();
            release_acc(ab ^ 1u);
          }
          if (jlast < 0) release_acc(ab);
          for (int j = 0; j < nblk; ++j) {
            const int b = cb[j];
            // TMEM columns of block j: D_re and D_im of its 128 columns.
            const uint32_t c_re = WIDE ? j * kBlk : ab * 256;
            const uint32_t c_im = WIDE ? 256 + j * kBlk : ab * 256 + kImCol;
#pragma unroll 1
            for (int piece = first_p[j]; piece <= last_p[j]; ++piece) {
              uint32_t vr[32], vi[32];
              ptx::tmem_ld_32x32b_x32(t_lanes + c_re + piece * 32, vr);
              ptx::tmem_ld_32x32b_x32(t_lanes + c_im + piece * 32, vi);
              if constexpr (kTmemSum) {
               if (!gfirst) {
                uint32_t sr[32], si[32];
                ptx::tmem_ld_32x32b_x32(t_lanes + 256 + piece * 32, sr);
                ptx::tmem_ld_32x32b_x32(t_lanes + 384 + piece * 32, si);
                ptx::tmem_wait_ld();
#pragma unroll
                for (int jj = 0; jj < 32; ++jj) {
                  vr[jj] = __float_as_uint(__uint_as_float(vr[jj]) + __uint_as_float(sr[jj]));
                  vi[jj] = __float_as_uint(__uint_as_float(vi[jj]) + __uint_as_float(si[jj]));
                }
               }
              }
              ptx::tmem_wait_ld();
              if (j == jlast && piece == last_p[j]) release_acc(ab);
              if (kTmemSum && !glast) {
                ptx::tmem_st_32x32b_x32(t_lanes + 256 + piece * 32, vr);
                ptx::tmem_st_32x32b_x32(t_lanes + 384 + piece * 32, vi);
                continue;
              }
              const int b0 = b * kBlk + piece * 32;
              const bool tr = b > k.a;  // a mirrored block
              if constexpr (IS_INT) {
                if (tr)
                  store_piece_tr<kWordInt>(vr, vi, p, f, a, b0, add, pol_out);
                else
                  store_piece<kWordInt>(vr, vi, p, f, a, b0, add, pol_out);
              } else {
                if (p.in_amax) scale_piece<FMT>(vr, vi, p, f, a, b0);
                // A drain that is both the first and the last of the running
                // sum (one chunk, or one chunk pair, without accumulation
                // across calls) only rounds to fp32: the plain store.
                if (p.acc64 && !(first && last_chunk && !p.accumulate)) {
                  if (tr)
                    store_piece_f64_tr(vr, vi, p, f, a, b0, first, last_chunk);
                  else
                    store_piece_f64(vr, vi, p, f, a, b0, first, last_chunk, pol_out);
                } else {
                  // With block sums on, this drain holds the whole
                  // integration: it overwrites `out` (a paired chunk's
                  // ch > 0 must not make it add).
                  const bool add_out = add && !p.acc64;
                  if (tr)
                    store_piece_tr<kWordFloat>(vr, vi, p, f, a, b0, add_out, pol_out);
                  else
                    store_piece<kWordFloat>(vr, vi, p, f, a, b0, add_out, pol_out);
                }
              }
            }
          }
          if (kTmemSum && !glast) ptx::tmem_wait_st();
          ++u;
        }
        kb0 = kb1;
      }
    }
  } else {
    // ---------------------------------------------------------- converters
    const int cw = warp - (2 + kNumEpiWarps);
    const uint32_t cbuf = sbase + C::kConvOff + cw * kConvBufBytes;
    static_assert((DT == 0) == (IN != kInFloat), "input form of the type");
    if constexpr (IN == kInTma) {
      converter_tma<FMT, MULTI, SHAPE>(bt, cbuf, conv_bar(cw), cw, lane, abort_flag);
    } else if constexpr (IN == kInWords) {
      bool even = true;
      for (int i = 0; i < bt.nsub; ++i) even = even && bt.sub[i].n % 2 == 0;
      if (even)
        converter_words<FMT, MULTI, SHAPE, true>(bt, cw, lane, abort_flag);
      else
        converter_words<FMT, MULTI, SHAPE, false>(bt, cw, lane, abort_flag);
    } else {
      if (bt.sub[0].tma_in) {
        converter_tma_float<DT, FMT, MULTI, SHAPE>(bt, cbuf, conv_bar(cw), cw, lane, abort_flag);
      } else {
        converter_direct<DT, FMT, MULTI, SHAPE>(bt, cw, lane, abort_flag);
      }
    }
  }

  // ------------------------------------------------------------- teardown
  ptx::tc_fence_before();
  __syncthreads();
  if constexpr (PAIR) ptx::cluster_sync();  // no SM still reads the other's shared memory or TMEM
  if (warp == 1) {
    ptx::tc_fence_after();
    if constexpr (PAIR) {
      ptx::tmem_dealloc_pair(tmem, kTmemCols);
    } else {
      ptx::tmem_dealloc(tmem, kTmemCols);
    }
  }
}

template <bool IS_INT, int DT, int FMT, bool MULTI, int IN>
__global__ void __launch_bounds__(threads_of<FMT, DT>(), 1) planar_kernel(const __grid_constant__ Batch bt) {
  planar_body<IS_INT, DT, FMT, MULTI, kShape128, IN>(bt);
}

// 128 x 256 items: one CTA, N = 256 MMAs.
template <bool IS_INT, int DT, int FMT, bool MULTI, int IN>
__global__ void __launch_bounds__(threads_of<FMT, DT>(), 1) planar_wide_kernel(const __grid_constant__ Batch bt) {
  if constexpr (FMT != kFmtHiLo) planar_body<IS_INT, DT, FMT, MULTI, kShapeWide, IN>(bt);
}

// CTA pairs: the cluster shape is part of the kernel, so no launch can run it
// without its peer.
template <bool IS_INT, int DT, int FMT, bool MULTI, int IN>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(threads_of<FMT, DT>(), 1)
    planar_pair_kernel(const __grid_constant__ Batch bt) {
  planar_body<IS_INT, DT, FMT, MULTI, kShapePair, IN>(bt);
}

}  // namespace
}  // namespace xc
