// xc_adjoint_tc.cu -- tensor-core adjoint of the float X-engine.
//
// For a real loss L, with grad_out scattered into G_f and H_f = G_f + G_f^H
// (xc_adjoint.cu), the input gradient is grad_x = conj(g) H_f (g x).  The
// gains fold into the matrix: H'_f = H_f diag(g), so per channel
//
//     grad_y[a][t] = sum_b H'[a][b] x[t][b],     grad_x = conj(g_a) grad_y,
//     grad_g[a]   += sum_t conj(x[t][a]) grad_y[a][t],
//
// a complex GEMM with M = a (inputs), N = t (samples), K = b (inputs).  It
// runs on tcgen05 in planar form:
//     Re = Hr Xr^T - Hi Xi^T,   Im = Hr Xi^T + Hi Xr^T,
// four 128 x 128 MMAs per 16-b step, the one of Hi Xi^T with negate-B.  (PTX
// orders back-to-back MMAs on an accumulator only when they have the same
// shape, so no 128 x 256 MMA, Hr [Xr Xi]^T, takes the place of two of them; it
// gave no time either.)  Operands are split into fp16 hi + lo parts after a
// power-of-two scale per row (input a of H', sample t of x, from its largest
// component), and each step runs three times (hi hi, lo hi, hi lo): about 22
// significant bits with fp32 accumulation over K = n.
//
// Kernels: operand formation, one pass over x and one over grad_out (H' is
// formed straight from it), into 8 KiB MMA-ready tiles ([8-row group]
// [8-column chunk][8 rows][8 fp16], the no-swizzle K-major layout); the GEMM,
// a persistent kernel over 128 x 128 (a, t) tiles with a bulk-copy producer
// warp, an MMA warp and eight epilogue warps that re-read x (nothing from the
// forward is stored).  A stage holds all eight tiles of 32 b (hi and lo, re and im, of
// both operands), 64 KiB for 24 MMAs: the three combinations share their
// operands' copies.
#include <cuda.h>
#include <cuda_fp16.h>

#include <algorithm>

#include "xc_launch.h"
#include "xc_ptx.cuh"

namespace xc {
namespace {

constexpr int kBlk = 128;  // rows per tile (a or t)
constexpr int kBK = 32;    // K (b) per tile
constexpr int kTile = kBlk * kBK * 2;
constexpr uint32_t kChunkStride = 8 * 16;  // between core matrices (8 rows x 16 B) adjacent in K
constexpr uint32_t kGroupStride = (kBK / 8) * kChunkStride;  // and in M / N
constexpr int kStages = 3;
constexpr int kOperand = 4 * kTile;  // (hi r, hi i, lo r, lo i)
constexpr int kStageBytes = 2 * kOperand;
constexpr int kEpiWarps = 8;  // two per TMEM lane quarter, half of the columns each
constexpr int kThreads = 32 * (2 + kEpiWarps);  // producer, MMA, epilogue
constexpr int kBarOff = kStages * kStageBytes;
constexpr int kNumBars = 2 * kStages + 5;
constexpr int kSmemBytes = kBarOff + kNumBars * 8 + 16 + 1024;
constexpr uint32_t kTmemCols = 512;  // 2 sets x (D_re, D_im)
constexpr uint32_t kIdesc = ptx::idesc_f16_f32(kBlk, kBlk);
constexpr uint32_t kIdescNegB = kIdesc | (1u << 14);

struct AdjGeom {
  Geometry g;
  int n;   // complex inputs N * P
  int na;  // 128-row blocks over a
  int nk;  // 32-column blocks over b (K)
  int nt;  // 128-row blocks over t
};

__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
  return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}

// Power-of-two scale exponent: max |v| 2^-e in [2^14, 2^15) (fp16 hi/lo),
// clamped so that products of two scales stay normal floats.
__device__ __forceinline__ int adj_scale_exp(unsigned bits) {
  const int E = static_cast<int>((bits >> 23) & 0xffu);
  if (E == 0) return 0;
  return max(-60, min(60, E - 127 - 14));
}
__device__ __forceinline__ float adj_exp2i(int e) { return __int_as_float((127 + e) << 23); }

// Byte offset of the operand tiles (hi r, hi i, lo r, lo i) of (channel f, row
// block rb, K block kb) in an operand buffer with nrb row blocks per channel.
__device__ __forceinline__ size_t tile_off(int f, int rb, int kb, int nrb, int nk) {
  return ((static_cast<size_t>(f) * nrb + rb) * nk + kb) * static_cast<size_t>(kOperand);
}

// hi + lo fp16 pairs of 8 scaled values: hi[4], lo[4] (two values per word).
__device__ __forceinline__ void split8(const float (&v)[8], uint32_t (&hi)[4], uint32_t (&lo)[4]) {
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const __half2 h = __floats2half2_rn(v[2 * k], v[2 * k + 1]);
    const __half2 l = __floats2half2_rn(v[2 * k] - __low2float(h), v[2 * k + 1] - __high2float(h));
    hi[k] = *reinterpret_cast<const uint32_t*>(&h);
    lo[k] = *reinterpret_cast<const uint32_t*>(&l);
  }
}

// Write the four 16-byte row chunks (hi re, hi im, lo re, lo im) of row r,
// 8-column chunk bc.
__device__ __forceinline__ void put_chunks(uint8_t* buf, int f, int r, int bc, int nrb, int nk,
                                           const float (&re)[8], const float (&im)[8]) {
  uint32_t rh[4], rl[4], ih[4], il[4];
  split8(re, rh, rl);
  split8(im, ih, il);
  uint8_t* o = buf + tile_off(f, r / kBlk, bc / (kBK / 8), nrb, nk) + (r % kBlk / 8) * kGroupStride +
               (bc % (kBK / 8)) * kChunkStride + (r % 8) * 16;
  *reinterpret_cast<uint4*>(o) = make_uint4(rh[0], rh[1], rh[2], rh[3]);
  *reinterpret_cast<uint4*>(o + kTile) = make_uint4(ih[0], ih[1], ih[2], ih[3]);
  *reinterpret_cast<uint4*>(o + 2 * kTile) = make_uint4(rl[0], rl[1], rl[2], rl[3]);
  *reinterpret_cast<uint4*>(o + 3 * kTile) = make_uint4(il[0], il[1], il[2], il[3]);
}

// Operand formation of 16 rows: thread (r, c) = (tid & 15, tid >> 4) takes
// chunks c, c + 16, ... of row r (consecutive threads take consecutive rows, so
// a warp writes four whole core matrices per plane).  load(chunk, v) gives the
// chunk's eight values.  Up to NC chunks per thread stay in registers between
// the row's maximum and its conversion: one pass over the input (rows of more
// chunks are loaded twice).  The row's exponent goes to exps[row].
constexpr int kFormRows = 16, kFormThreads = 256, kFormCols = kFormThreads / kFormRows;
template <int NC, typename Load>
__device__ __forceinline__ void form_rows(Load load, int row, int f, uint8_t* buf, int* exps, int nrb, int nk) {
  __shared__ unsigned smax[kFormRows];
  const int r = threadIdx.x % kFormRows, c = threadIdx.x / kFormRows;
  const int nch = nk * (kBK / 8);
  if (threadIdx.x < kFormRows) smax[threadIdx.x] = 0;
  __syncthreads();
  float2 v[NC][8];
  float m = 0.f;
  const bool fits = nch <= NC * kFormCols;
  if (fits) {
#pragma unroll
    for (int i = 0; i < NC; ++i)
      if (c + i * kFormCols < nch) load(c + i * kFormCols, v[i]);
#pragma unroll
    for (int i = 0; i < NC; ++i)
      if (c + i * kFormCols < nch)
#pragma unroll
        for (int j = 0; j < 8; ++j) m = fmaxf(m, fmaxf(fabsf(v[i][j].x), fabsf(v[i][j].y)));
  } else {
    for (int ch = c; ch < nch; ch += kFormCols) {
      load(ch, v[0]);
#pragma unroll
      for (int j = 0; j < 8; ++j) m = fmaxf(m, fmaxf(fabsf(v[0][j].x), fabsf(v[0][j].y)));
    }
  }
  // (The lanes l and l + 16 of a warp have the same row.)
  m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, 16));
  if ((threadIdx.x & 16) == 0) atomicMax(&smax[r], __float_as_uint(m));
  __syncthreads();
  const int e = adj_scale_exp(smax[r]);
  if (c == 0) exps[row] = e;
  const float s = adj_exp2i(-e);
  auto put = [&](int ch, const float2 (&w)[8]) {
    float re[8], im[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      re[j] = w[j].x * s;
      im[j] = w[j].y * s;
    }
    put_chunks(buf, f, row, ch, nrb, nk, re, im);
  };
  if (fits) {
#pragma unroll
    for (int i = 0; i < NC; ++i)
      if (c + i * kFormCols < nch) put(c + i * kFormCols, v[i]);
  } else {
    for (int ch = c; ch < nch; ch += kFormCols) {
      load(ch, v[0]);
      put(ch, v[0]);
    }
  }
}

// A operand: H'_f = H_f diag(g) with H_f = G_f + G_f^H, rows a (padded to na *
// 128), K = b (padded to nk * 32), straight from the packed grad_out (each
// off-diagonal entry of it is read twice, through L2): 60 us at 64 channels of
// 512 inputs (182 us by way of H in memory and a pass for its maximum).
template <int NC>
__global__ void __launch_bounds__(kFormThreads) adj_form_h(const float2* __restrict__ grad_out,
                                                           const float2* __restrict__ gains,
                                                           uint8_t* __restrict__ At, int* __restrict__ exps,
                                                           AdjGeom G) {
  const int f = blockIdx.y, a = blockIdx.x * kFormRows + threadIdx.x % kFormRows;
  const int P = G.g.P, PP = P * P, sh = P - 1;  // P is 1 or 2
  const int sa = a >> sh, pa = a & sh;
  const float2* go = grad_out + static_cast<int64_t>(f) * G.g.NB * PP;
  const float2* row = go + static_cast<int64_t>(sa) * (sa + 1) / 2 * PP + pa * P;
  auto load = [&](int ch, float2 (&v)[8]) {
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const int b = ch * 8 + j, sb = b >> sh, pb = b & sh;
      float2 h = make_float2(0.f, 0.f);
      if (a < G.n && b < G.n) {
        if (sb <= sa) h = row[sb * PP + pb];  // G[a][b]
        if (sb >= sa) {                       // conj(G[b][a])
          const float2 w = go[(static_cast<int64_t>(sb) * (sb + 1) / 2 + sa) * PP + pb * P + pa];
          h.x += w.x;
          h.y -= w.y;
        }
        if (gains) h = cmul(h, gains[b]);
      }
      v[j] = h;
    }
  };
  form_rows<NC>(load, a, f, At, exps + static_cast<size_t>(f) * G.na * kBlk, G.na, G.nk);
}

// B operand: x tiles, rows t (padded to nt * 128), K = b.  Bound by its one
// read of x and the same bytes written (hi and lo halves): 2.1 GB in 308 us on
// 256 stations x 2 pols, F=64, T=4096 (a pass for one maximum per channel and
// one to form the tiles took 241 + 481 us).
template <int NC>
__global__ void __launch_bounds__(kFormThreads) adj_form_x(const float2* __restrict__ x, uint8_t* __restrict__ Bt,
                                                           int* __restrict__ exps, AdjGeom G) {
  const int f = blockIdx.y, t = blockIdx.x * kFormRows + threadIdx.x % kFormRows;
  const float2* row = x + (static_cast<int64_t>(t) * G.g.F + f) * G.n;
  const bool vec = G.n % 2 == 0;  // rows start on 16 bytes
  auto load = [&](int ch, float2 (&v)[8]) {
    if (t < G.g.T && vec && ch * 8 + 8 <= G.n) {
      const float4* q = reinterpret_cast<const float4*>(row + ch * 8);
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const float4 w = __ldg(q + j);
        v[2 * j] = make_float2(w.x, w.y);
        v[2 * j + 1] = make_float2(w.z, w.w);
      }
    } else {
#pragma unroll
      for (int j = 0; j < 8; ++j)
        v[j] = t < G.g.T && ch * 8 + j < G.n ? __ldg(row + ch * 8 + j) : make_float2(0.f, 0.f);
    }
  };
  form_rows<NC>(load, t, f, Bt, exps + static_cast<size_t>(f) * G.nt * kBlk, G.nt, G.nk);
}

struct AdjParams {
  AdjGeom G;
  const uint8_t* At;
  const uint8_t* Bt;
  const int* exp_h;  // [F][na * 128] row exponents of H'
  const int* exp_x;  // [F][nt * 128] of x
  const float2* x;
  const float2* gains;
  float2* grad_x;
  double* grad_g;  // running sums, rounded to the caller's fp32 at the end
  unsigned long long timeout_ns;
  int* status;
};

// Persistent GEMM: CTA i takes tiles i, i + grid, ... in (channel, t block,
// a block) order with the a block fastest, so the CTAs working at one time
// share their x tiles (and a channel's H' tiles) through L2.  The stage ring
// runs on across tiles and the accumulator is double-buffered in TMEM: the
// epilogue of one tile overlaps the MMAs of the next.
__global__ void __launch_bounds__(kThreads, 1) adj_gemm_tc(const AdjParams P) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                             ~static_cast<uintptr_t>(1023));
  const uint32_t sbase = ptx::smem_u32(smem);
  const uint32_t bar0 = sbase + kBarOff;
  auto full_bar = [&](int s) { return bar0 + 8u * s; };
  auto empty_bar = [&](int s) { return bar0 + 8u * (kStages + s); };
  auto accf_bar = [&](int b) { return bar0 + 8u * (2 * kStages + b); };
  auto acce_bar = [&](int b) { return bar0 + 8u * (2 * kStages + 2 + b); };
  const uint32_t drain_bar = bar0 + 8u * (2 * kStages + 4);
  uint32_t* tmem_holder = reinterpret_cast<uint32_t*>(smem + kBarOff + kNumBars * 8);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_holder + 1);
  const int warp = __shfl_sync(0xffffffffu, static_cast<int>(threadIdx.x >> 5), 0);  // (known uniform)
  const int lane = threadIdx.x & 31;
  const AdjGeom& G = P.G;
  const long long ntiles = static_cast<long long>(G.g.F) * G.nt * G.na;
  auto tile_of = [&](long long it, int* f, int* tb, int* ab) {
    *ab = static_cast<int>(it % G.na);
    const long long r = it / G.na;
    *tb = static_cast<int>(r % G.nt);
    *f = static_cast<int>(r / G.nt);
  };

  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) {
      ptx::mbar_init(full_bar(s), 1);
      ptx::mbar_init(empty_bar(s), 1);
    }
    for (int b = 0; b < 2; ++b) {
      ptx::mbar_init(accf_bar(b), 1);
      ptx::mbar_init(acce_bar(b), kEpiWarps);
    }
    ptx::mbar_init(drain_bar, 1);
    *abort_flag = 0;
    ptx::fence_mbar_init();
    ptx::fence_proxy_async_smem();
  }
  if (warp == 1) {
    ptx::tmem_alloc(ptx::smem_u32(tmem_holder), kTmemCols);
    ptx::tmem_relinquish();
  }
  ptx::tc_fence_before();
  __syncthreads();
  ptx::tc_fence_after();
  const uint32_t tmem = *tmem_holder;
  const ptx::WaitCtl wc{P.timeout_ns, P.status, abort_flag};

  if (warp == 0) {
    if (lane == 0) {
      int issued_phase[kStages];
      for (int s = 0; s < kStages; ++s) issued_phase[s] = -1;
      bool ok = true;
      int stage = 0;  // the stage ring runs on across tiles
      uint32_t phase = 0;
      for (long long it = blockIdx.x; ok && it < ntiles; it += gridDim.x) {
        int f, tb, ab;
        tile_of(it, &f, &tb, &ab);
        for (int kb = 0; kb < G.nk; ++kb) {
          if (!ptx::wait_bounded(empty_bar(stage), phase ^ 1u, wc)) {
            ok = false;
            break;
          }
          const uint32_t dst = sbase + stage * kStageBytes;
          const uint32_t fb = full_bar(stage);
          ptx::mbar_arrive_expect_tx(fb, kStageBytes);
          ptx::bulk_load(dst, P.At + tile_off(f, ab, kb, G.na, G.nk), kOperand, fb);
          ptx::bulk_load(dst + kOperand, P.Bt + tile_off(f, tb, kb, G.nt, G.nk), kOperand, fb);
          issued_phase[stage] = static_cast<int>(phase);
          if (++stage == kStages) {
            stage = 0;
            phase ^= 1u;
          }
        }
      }
      if (!ok) {
        for (int s = 0; s < kStages; ++s) {
          if (issued_phase[s] < 0) continue;
          const uint64_t t0 = ptx::globaltimer();
          while (!ptx::mbar_try_wait(full_bar(s), static_cast<uint32_t>(issued_phase[s])) &&
                 ptx::globaltimer() - t0 < P.timeout_ns) {
          }
        }
      }
    }
  } else if (warp == 1) {
    // The whole warp walks the stages (loop state and descriptors stay
    // warp-uniform); one elected lane issues.
    const bool issuer = ptx::elect_one();
    bool ok = true;
    int stage = 0;
    uint32_t phase = 0;
    uint32_t u = 0;  // tiles done by this CTA
    const uint64_t desc0 = ptx::interleave_kmajor_desc(sbase, kChunkStride, kGroupStride);
    constexpr uint64_t kT = kTile >> 4;
    for (long long it = blockIdx.x; ok && it < ntiles; it += gridDim.x, ++u) {
      const uint32_t ab = u & 1u, ap = (u >> 1) & 1u;
      bool got = ptx::wait_bounded(acce_bar(ab), ap ^ 1u, wc);
      if (!__all_sync(0xffffffffu, got)) {
        ok = false;
        break;
      }
      const uint32_t d_re = tmem + ab * 256, d_im = d_re + 128;
      for (int kb = 0; kb < G.nk; ++kb) {
        got = ptx::wait_bounded(full_bar(stage), phase, wc);
        if (!__all_sync(0xffffffffu, got)) {
          ok = false;
          break;
        }
        ptx::tc_fence_after();
        const uint64_t dh = desc0 + static_cast<uint64_t>(stage) * (kStageBytes >> 4), dx = dh + (kOperand >> 4);
        if (issuer) {
#pragma unroll
          for (int k = 0; k < kBK / 16; ++k) {
#pragma unroll
            for (int j = 0; j < 3; ++j) {  // (hi, hi), (lo, hi), (hi, lo)
              const uint64_t ko = static_cast<uint64_t>(k * 2 * kChunkStride) >> 4;
              const uint64_t dhr = dh + (j == 1 ? 2 * kT : 0) + ko, dhi = dhr + kT;
              const uint64_t dxr = dx + (j == 2 ? 2 * kT : 0) + ko, dxi = dxr + kT;
              const uint32_t acc = (kb > 0 || k > 0 || j > 0) ? 1u : 0u;
              ptx::mma_f16_ss(d_re, dhr, dxr, kIdesc, acc);     // Re += Hr Xr^T
              ptx::mma_f16_ss(d_re, dhi, dxi, kIdescNegB, 1u);  // Re -= Hi Xi^T
              ptx::mma_f16_ss(d_im, dhr, dxi, kIdesc, acc);     // Im += Hr Xi^T
              ptx::mma_f16_ss(d_im, dhi, dxr, kIdesc, 1u);      // Im += Hi Xr^T
            }
          }
          ptx::mma_commit(empty_bar(stage));
        }
        if (++stage == kStages) {
          stage = 0;
          phase ^= 1u;
        }
      }
      if (ok && issuer) ptx::mma_commit(accf_bar(ab));
    }
    if (!ok && issuer) {
      // The MMAs issued so far complete before TMEM is freed (bounded).
      ptx::mma_commit(drain_bar);
      const uint64_t t0 = ptx::globaltimer();
      while (!ptx::mbar_try_wait(drain_bar, 0) && ptx::globaltimer() - t0 < P.timeout_ns) {
      }
    }
    __syncwarp();
  } else {
    // Epilogue: warp q owns TMEM lanes 32q..32q+31 = rows a of the tile.  Its
    // reads of x and writes of grad_x are latency-bound: with one warp per lane
    // quarter a tile takes 19.8 us, with two 17.6 us (its MMAs alone 13 us;
    // 256 stations x 2 pols, F=64, T=4096: 1065 and 947 us).
    const int q = warp & 3;
    constexpr int kPieces = kBlk / 32 * 4 / kEpiWarps;  // 32-column pieces per warp
    const int piece0 = (warp - 2) / 4 * kPieces;
    const uint32_t t_lanes = tmem + (static_cast<uint32_t>(q * 32) << 16);
    uint32_t u = 0;
    for (long long it = blockIdx.x; it < ntiles; it += gridDim.x, ++u) {
      int f, tb, abk;
      tile_of(it, &f, &tb, &abk);
      const uint32_t ab = u & 1u, ap = (u >> 1) & 1u;
      const bool got = ptx::wait_bounded(accf_bar(ab), ap, wc);
      if (!__all_sync(0xffffffffu, got)) break;
      ptx::tc_fence_after();
      const int a = abk * kBlk + q * 32 + lane;
      const bool row_ok = a < G.n;
      const int eh = P.exp_h[static_cast<size_t>(f) * G.na * kBlk + a];
      const int* ex = P.exp_x + (static_cast<size_t>(f) * G.nt + tb) * kBlk;
      const float2 ga = (P.gains && row_ok) ? P.gains[a] : make_float2(1.f, 0.f);
      const float2 cga = make_float2(ga.x, -ga.y);
      float2 gg = make_float2(0.f, 0.f);
#pragma unroll 1
      for (int piece = piece0; piece < piece0 + kPieces; ++piece) {
        uint32_t vr[32], vi[32];
        ptx::tmem_ld_32x32b_x32(t_lanes + ab * 256 + piece * 32, vr);
        ptx::tmem_ld_32x32b_x32(t_lanes + ab * 256 + 128 + piece * 32, vi);
        ptx::tmem_wait_ld();
        if (piece == piece0 + kPieces - 1) {
          ptx::tc_fence_before();
          __syncwarp();
          if (lane == 0) ptx::mbar_arrive(acce_bar(ab));
        }
        if (!row_ok) continue;
        // All 32 samples of x first (the compiler may not move these loads
        // above the grad_x stores), then grad_x and the grad_g terms.
        const int t0 = tb * kBlk + piece * 32;
        const size_t step = static_cast<size_t>(G.g.F) * G.n;
        const size_t idx0 = (static_cast<size_t>(t0) * G.g.F + f) * G.n + a;
        float2 xv[32];
#pragma unroll
        for (int j = 0; j < 32; ++j)
          xv[j] = t0 + j < G.g.T ? __ldcs(P.x + idx0 + j * step) : make_float2(0.f, 0.f);
#pragma unroll
        for (int j = 0; j < 32; ++j) {
          if (t0 + j >= G.g.T) continue;
          const float sc = adj_exp2i(eh + __ldg(ex + piece * 32 + j));  // (one address for the warp)
          const float2 gy = make_float2(__uint_as_float(vr[j]) * sc, __uint_as_float(vi[j]) * sc);
          __stcs(P.grad_x + idx0 + j * step, cmul(cga, gy));
          gg.x += xv[j].x * gy.x + xv[j].y * gy.y;  // conj(x) gy
          gg.y += xv[j].x * gy.y - xv[j].y * gy.x;
        }
      }
      if (row_ok && P.grad_g) {
        atomicAdd(P.grad_g + 2 * a, static_cast<double>(gg.x));
        atomicAdd(P.grad_g + 2 * a + 1, static_cast<double>(gg.y));
      }
    }
  }
  ptx::tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    ptx::tc_fence_after();
    ptx::tmem_dealloc(tmem, kTmemCols);
  }
}

// The gain gradient's sums over all tiles, added in float64 (fp32 partial sums
// of 64 samples each).
__global__ void adj_round_gains(const double* __restrict__ sums, float* __restrict__ grad_g, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) grad_g[i] = static_cast<float>(sums[i]);
}

AdjGeom adj_geom(const Geometry& g) {
  AdjGeom G;
  G.g = g;
  G.n = g.N * g.P;
  G.na = (G.n + kBlk - 1) / kBlk;
  G.nk = (G.n + kBK - 1) / kBK;
  G.nt = (g.T + kBlk - 1) / kBlk;
  return G;
}

}  // namespace

size_t adjoint_tc_workspace_bytes(const Geometry& g) {
  const AdjGeom G = adj_geom(g);
  const size_t per_rb = static_cast<size_t>(G.nk) * kOperand + kBlk * sizeof(int);  // tiles, row exponents
  return static_cast<size_t>(g.F) * (G.na + G.nt) * per_rb + 2 * sizeof(double) * G.n;
}

cudaError_t launch_adjoint_tc(const void* grad_out, const void* in, const void* gains, void* grad_in,
                              float* grad_g, void* tc_ws, const Geometry& g, unsigned long long timeout_ns,
                              int* status, cudaStream_t s) {
  const AdjGeom G = adj_geom(g);
  if (G.n == 0 || g.F == 0 || g.T == 0) return cudaSuccess;
  uint8_t* At = static_cast<uint8_t*>(tc_ws);
  const size_t per_rb = static_cast<size_t>(G.nk) * kOperand;
  uint8_t* Bt = At + static_cast<size_t>(g.F) * G.na * per_rb;
  int* exp_h = reinterpret_cast<int*>(Bt + static_cast<size_t>(g.F) * G.nt * per_rb);
  int* exp_x = exp_h + static_cast<size_t>(g.F) * G.na * kBlk;
  const float2* go = static_cast<const float2*>(grad_out);
  const float2* x = static_cast<const float2*>(in);
  const float2* gn = static_cast<const float2*>(gains);
  cudaError_t e = cudaSuccess;
  double* sums = reinterpret_cast<double*>(exp_x + static_cast<size_t>(g.F) * G.nt * kBlk);
  if (grad_g) e = cudaMemsetAsync(sums, 0, sizeof(double) * 2 * G.n, s);
  if (e != cudaSuccess) return e;
  // Chunks per thread: four (rows of up to 512 inputs in one pass) or one.
  const dim3 gh(G.na * (kBlk / kFormRows), g.F), gx(G.nt * (kBlk / kFormRows), g.F);
  if (G.nk * (kBK / 8) > kFormCols) {
    adj_form_h<4><<<gh, kFormThreads, 0, s>>>(go, gn, At, exp_h, G);
    adj_form_x<4><<<gx, kFormThreads, 0, s>>>(x, Bt, exp_x, G);
  } else {
    adj_form_h<1><<<gh, kFormThreads, 0, s>>>(go, gn, At, exp_h, G);
    adj_form_x<1><<<gx, kFormThreads, 0, s>>>(x, Bt, exp_x, G);
  }
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  e = cudaFuncSetAttribute(adj_gemm_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes);
  if (e != cudaSuccess) return e;
  AdjParams P;
  P.G = G;
  P.At = At;
  P.Bt = Bt;
  P.exp_h = exp_h;
  P.exp_x = exp_x;
  P.x = x;
  P.gains = gn;
  P.grad_x = static_cast<float2*>(grad_in);
  P.grad_g = grad_g ? sums : nullptr;
  P.timeout_ns = timeout_ns;
  P.status = status;
  int dev = 0, sms = 0;
  e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  const long long ntiles = static_cast<long long>(g.F) * G.nt * G.na;
  adj_gemm_tc<<<static_cast<unsigned>(std::min<long long>(ntiles, sms)), kThreads, kSmemBytes, s>>>(P);
  if (grad_g) adj_round_gains<<<(2 * G.n + 255) / 256, 256, 0, s>>>(sums, grad_g, 2 * G.n);
  return cudaGetLastError();
}

}  // namespace xc
