// xc_planar.cu -- host side of the planar tensor-core X-engine (the kernel
// template is xc_planar_kernel.cuh): the single-CTA instantiations, the
// float scale pre-pass, the kernel parameter block and the launch (single CTAs,
// or CTA pairs from xc_planar_pair.cu).  Its sizes are decided in
// xc_planar_plan.h.
#include "xc_planar_kernel.cuh"

namespace xc {

// The CTA-pair and 128 x 256 instantiations live in xc_planar_pair.cu and
// xc_planar_wide.cu (compiled in parallel with this file).
const void* planar_pair_select(int in_dtype, int fmt, bool multi);
const void* planar_wide_select(int in_dtype, int fmt, bool multi);
// 8-bit rows that TMA cannot stride, every shape (xc_planar_words.cu).
const void* planar_words_select(int shape, int fmt, bool multi);

static_assert(kShape128 == kPlanar128 && kShapePair == kPlanarPair && kShapeWide == kPlanarWide,
              "tile shape codes");
static_assert(kFmtF16 == XC_PREC_FP16 && kFmtHiLo == XC_PREC_HILO && kFmtF8 == XC_PREC_FP8 && kBlk == kPlanarBlk,
              "xc_planar_plan.h counts in the kernel's formats and blocks");

namespace {

template <bool IS_INT, int DT, int FMT, bool MULTI = false>
const void* kernel_of() {
  return reinterpret_cast<const void*>(planar_kernel<IS_INT, DT, FMT, MULTI, IS_INT ? kInTma : kInFloat>);
}

// Batches of several subarrays take 8-bit input.
const void* select_kernel(int in_dtype, int fmt, bool multi) {
  if (in_dtype == 0) {
    if (fmt == kFmtF8) return multi ? nullptr : kernel_of<true, 0, kFmtF8>();
    return multi ? kernel_of<true, 0, kFmtF16, true>() : kernel_of<true, 0, kFmtF16>();
  }
  if (multi) return nullptr;
  if (in_dtype != 1 && in_dtype != 2) return nullptr;
  const bool h = in_dtype == 1;
  switch (fmt) {
    case kFmtF16: return h ? kernel_of<false, 1, kFmtF16>() : kernel_of<false, 2, kFmtF16>();
    case kFmtHiLo: return h ? kernel_of<false, 1, kFmtHiLo>() : kernel_of<false, 2, kFmtHiLo>();
    case kFmtF8: return h ? kernel_of<false, 1, kFmtF8>() : kernel_of<false, 2, kFmtF8>();
    default: return nullptr;
  }
}

// Scale pre-pass for float input: amax[f][a] = max over t of the largest
// component of g_a x_a(t) (fp32 bits; non-negative floats order as
// unsigned integers).  Bound by the one read of the input: a thread keeps
// eight 16-byte loads in flight (VEC = 2 complex fp32 or 4 complex fp16
// inputs; VEC = 1 when a row is not a multiple of 16 bytes).  A block takes
// kAmaxIter x `rows` samples of one channel, `rows` of them side by side when
// a row has fewer than 128 vectors.  On 512 stations x 2 pols, F=60, T=2048,
// fp32 (1.0 GB): 138 us (291 us with one 8-byte load per input and sample).
constexpr int kAmaxThreads = 128, kAmaxIter = 64;
template <int DT, int VEC>
__global__ void __launch_bounds__(kAmaxThreads) input_amax_kernel(const void* __restrict__ in,
                                                                  const float2* __restrict__ gains,
                                                                  unsigned* __restrict__ amax, Geometry g,
                                                                  int n, int gain_n, int rows) {
  const int nv = n / VEC;  // vectors of a row
  const int r = rows > 1 ? threadIdx.x / nv : 0;
  const int v = rows > 1 ? threadIdx.x - r * nv : blockIdx.x * kAmaxThreads + threadIdx.x;
  const int f = blockIdx.y;
  if (v >= nv || r >= rows) return;
  const int a = v * VEC;
  const int t0 = blockIdx.z * kAmaxIter * rows + r;
  const int t1 = min(g.T, static_cast<int>(blockIdx.z + 1) * kAmaxIter * rows);
  float2 ga[VEC];
  float m[VEC];
#pragma unroll
  for (int i = 0; i < VEC; ++i) {
    ga[i] = gains ? gains[(a + i) % gain_n] : make_float2(1.f, 0.f);
    m[i] = 0.f;
  }
  constexpr int kBytes = (DT == 1 ? 4 : 8) * VEC;
  using Raw = typename std::conditional<kBytes == 16, uint4, typename std::conditional<kBytes == 8, uint2, unsigned>::type>::type;
  const Raw* p = reinterpret_cast<const Raw*>(in) + (static_cast<int64_t>(t0) * g.F + f) * nv + v;
  const int64_t step = static_cast<int64_t>(rows) * g.F * nv;
  auto use = [&](const Raw& raw) {
#pragma unroll
    for (int i = 0; i < VEC; ++i) {
      float2 x;
      if constexpr (DT == 1) {
        x = __half22float2(reinterpret_cast<const __half2*>(&raw)[i]);
      } else {
        x = reinterpret_cast<const float2*>(&raw)[i];
      }
      if (gains) x = make_float2(ga[i].x * x.x - ga[i].y * x.y, ga[i].x * x.y + ga[i].y * x.x);
      m[i] = fmaxf(m[i], fmaxf(fabsf(x.x), fabsf(x.y)));
    }
  };
  int t = t0;
  for (; t + 7 * rows < t1; t += 8 * rows, p += 8 * step) {
    Raw w[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) w[i] = __ldg(p + i * step);
#pragma unroll
    for (int i = 0; i < 8; ++i) use(w[i]);
  }
  for (; t < t1; t += rows, p += step) use(__ldg(p));
#pragma unroll
  for (int i = 0; i < VEC; ++i) atomicMax(amax + static_cast<int64_t>(f) * n + a + i, __float_as_uint(m[i]));
}

template <int DT, int VEC>
cudaError_t launch_amax(const XeLaunch& L, int n, cudaStream_t s) {
  const int nv = n / VEC;
  const int rows = std::max(1, kAmaxThreads / nv);
  const dim3 grid(rows > 1 ? 1 : (nv + kAmaxThreads - 1) / kAmaxThreads, L.g.F,
                  (L.g.T + kAmaxIter * rows - 1) / (kAmaxIter * rows));
  if (grid.z > 65535u) return cudaErrorInvalidConfiguration;
  input_amax_kernel<DT, VEC><<<grid, kAmaxThreads, 0, s>>>(L.in, static_cast<const float2*>(L.gains), L.in_amax,
                                                          L.g, n, n / std::max(1, L.pack), rows);
  return cudaGetLastError();
}

// fast_div's magic of a divisor (0 for a divisor of 0, which nothing divides by).
unsigned div_magic(int d) {
  return d <= 0 ? 0u : d == 1 ? 0xffffffffu : static_cast<unsigned>((1ull << 32) / static_cast<unsigned>(d));
}

// Kernel parameters of one subarray.
Params sub_params(const XeLaunch& L, int shape) {
  Params p;
  p.g = L.g;
  p.n = L.g.N * L.g.P;
  p.in = L.in;
  p.out = L.out;
  p.accumulate = L.accumulate;
  p.nib = (p.n + kBlk - 1) / kBlk;
  p.ntiles = p.nib * (p.nib + 1) / 2;
  p.ipc = shape != kShape128 ? pair_items(p.nib) : p.ntiles;
  p.nitems = static_cast<long long>(p.ipc) * L.g.F;
  p.nkb = L.g.Tp / kBK;
  p.is_int = L.in_dtype == 0 ? 1 : 0;
  const int fmt = p.is_int ? (L.fmt == kFmtF8 ? kFmtF8 : kFmtF16) : L.fmt;
  p.seg_kb = std::max(1, L.ring_seg_kb);
  p.nseg = (p.nkb + p.seg_kb - 1) / p.seg_kb;
  p.nkt = (fmt == kFmtHiLo ? 2 : 1) * p.seg_kb;
  p.amax = L.amax;
  p.gains = static_cast<const float2*>(L.gains);
  p.in_amax = p.is_int ? nullptr : L.in_amax;
  p.acc64 = p.is_int ? nullptr : L.acc64;
  p.f_chunk_kb = p.nkb;
  if (p.acc64 && L.f64_block > 0) p.f_chunk_kb = std::max(1, std::min(p.nkb, L.f64_block / kBK));
  p.ring = static_cast<uint8_t*>(L.ring);
  p.ring_slots = L.ring_slots;
  p.ready = L.counters;
  p.done = L.counters + L.ring_slots;
  p.seg_units = (p.n + 63) / 64 * p.seg_kb;  // (half blocks with no input are left as they are)
  p.mag_kb = div_magic(p.seg_kb);
  p.mag_slots = div_magic(p.ring_slots);
  p.tma_in = 0;
  p.timeout_ns = L.timeout_ns;
  p.status = L.status;
  p.test_no_publish = L.test_no_publish;
  p.pack = std::max(1, L.pack);
  p.Nr = L.g.N / p.pack;
  p.NBr = static_cast<int64_t>(p.Nr) * (p.Nr + 1) / 2;
  p.gain_n = p.Nr * L.g.P;
  return p;
}

}  // namespace

cudaError_t planar_prepare(const XeLaunch* subs, const CUtensorMap* const* maps, int nsub,
                           PlanarKernel* k, int shape) {
  if (nsub < 1 || nsub > kMaxSub || !subs || !k) return cudaErrorInvalidValue;
  const int dt = subs[0].in_dtype;
  // 8-bit input: fp16 operands, or e4m3 when asked for (exact for |x| <= 16).
  auto fmt_of = [](const XeLaunch& L) {
    return L.in_dtype == 0 ? (L.fmt == kFmtF8 ? kFmtF8 : kFmtF16) : L.fmt;
  };
  const int fmt = fmt_of(subs[0]);
  Batch* b = reinterpret_cast<Batch*>(k->args);
  memset(b, 0, sizeof(Batch));
  b->nsub = nsub;
  bool all_tma = true;
  for (int i = 0; i < nsub; ++i) {
    if (subs[i].in_dtype != dt || fmt_of(subs[i]) != fmt) return cudaErrorInvalidValue;
    b->sub[i] = sub_params(subs[i], shape);
    if (subs[i].ring_slots < 1 || subs[i].ring_slots > subs[i].counter_slots) return cudaErrorInvalidValue;
    if (dt == 0 && static_cast<int64_t>(subs[i].g.F) * b->sub[i].nseg > subs[i].amax_words) return cudaErrorInvalidValue;
    if (maps && maps[i]) {
      b->maps[i] = *maps[i];
    } else {
      all_tma = false;
    }
    b->item_base[i + 1] = b->item_base[i] + (b->sub[i].nkb > 0 ? b->sub[i].nitems : 0);
    b->unit_base[i + 1] = b->unit_base[i] +
                          static_cast<long long>(subs[i].g.F) * b->sub[i].nseg * b->sub[i].seg_units;
  }
  for (int i = 0; i < nsub; ++i) b->sub[i].tma_in = all_tma ? 1 : 0;
  const int conv = (fmt == kFmtF8 && dt == 0) ? conv_warps<kFmtF8, 0>() : conv_warps<kFmtF16, 0>();
  const bool pair = shape == kShapePair;
  const bool words = dt == 0 && !all_tma;
  switch (words ? -1 : shape) {
    case -1: k->func = planar_words_select(shape, fmt, nsub > 1); break;
    case kShape128: k->func = select_kernel(dt, fmt, nsub > 1); break;
    case kShapePair: k->func = planar_pair_select(dt, fmt, nsub > 1); break;
    case kShapeWide: k->func = planar_wide_select(dt, fmt, nsub > 1); break;
    default: k->func = nullptr;
  }
  if (!k->func) return cudaErrorInvalidValue;
  const bool f8 = fmt == kFmtF8 && dt == 0;  // the e4m3 plan of 8-bit input
  k->block = f8 ? threads_of<kFmtF8, 0>() : threads_of<kFmtF16, 0>();
  k->smem = shape == kShapePair
                ? (f8 ? Cfg<kShapePair, kFmtF8, 0>::kSmemBytes : Cfg<kShapePair, kFmtF16, 0>::kSmemBytes)
                : (shape == kShapeWide
                       ? (f8 ? Cfg<kShapeWide, kFmtF8, 0>::kSmemBytes : Cfg<kShapeWide, kFmtF16, 0>::kSmemBytes)
                       : (f8 ? Cfg<kShape128, kFmtF8, 0>::kSmemBytes : Cfg<kShape128, kFmtF16, 0>::kSmemBytes));
  k->shape = shape;
  cudaError_t e = cudaFuncSetAttribute(k->func, cudaFuncAttributeMaxDynamicSharedMemorySize, k->smem);
  if (e != cudaSuccess) return e;
  // Every CTA must be resident at once: the operand ring couples them.
  const long long items = b->item_base[nsub];
  if (pair) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(static_cast<unsigned>(std::max(2, subs[0].grid & ~1)));
    cfg.blockDim = dim3(static_cast<unsigned>(k->block));
    cfg.dynamicSmemBytes = static_cast<size_t>(k->smem);
    int clusters = 0;
    e = cudaOccupancyMaxActiveClusters(&clusters, k->func, &cfg);
    if (e != cudaSuccess) return e;
    if (clusters < 1) return cudaErrorInvalidConfiguration;
    const long long ncl = std::min<long long>({static_cast<long long>(clusters), subs[0].grid / 2, items});
    k->grid = static_cast<int>(2 * ncl);
  } else {
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k->func, k->block, static_cast<size_t>(k->smem));
    if (e != cudaSuccess) return e;
    if (per_sm < 1) return cudaErrorInvalidConfiguration;
    const long long resident = static_cast<long long>(per_sm) * subs[0].grid;
    k->grid = static_cast<int>(std::min<long long>({items, static_cast<long long>(subs[0].grid), resident}));
  }
  // Runs of two units once every converter warp has eight or more to do (and a
  // segment is an even number of units), of one below (2 stations x 1 pol, F=11,
  // T=102: one CTA, 24 -> 17 us).  Then a warp's step from one run to its next,
  // for its incremental unit numbers.
  const long long workers = static_cast<long long>(k->grid) * conv;
  int run = b->unit_base[nsub] >= 8 * workers ? kUnitRun : 1;
  for (int i = 0; i < nsub; ++i)
    if (b->sub[i].seg_units % kUnitRun != 0) run = 1;
  const long long step = workers * run;
  for (int i = 0; i < nsub; ++i) {
    Params& p = b->sub[i];
    p.run = run;
    p.step_seg = static_cast<int>(step / p.seg_units);
    p.step_rem = static_cast<int>(step % p.seg_units);
    p.step_gen = p.step_seg / p.ring_slots;
    p.step_slot = p.step_seg % p.ring_slots;
    const int item_step = pair ? k->grid / 2 : k->grid;
    p.wave = planar_wave(item_step, p.ipc, p.ring_slots, p.g.F);
    if (p.ipc > item_step && p.ring_slots < p.nseg) return cudaErrorInvalidConfiguration;
    p.wave_segs = p.wave * p.nseg;
    p.wave_full = p.g.F / p.wave;
    p.wave_last = p.g.F - p.wave_full * p.wave;
    p.last_base = p.wave_full * p.wave_segs;
    p.mag_wave = div_magic(p.wave);
    p.mag_wsegs = div_magic(p.wave_segs);
    p.mag_last = div_magic(p.wave_last);
    p.it_step_f = item_step / p.ipc;
    p.it_step_i = item_step % p.ipc;
  }
  return cudaSuccess;
}

cudaError_t planar_setup(const XeLaunch* subs, int nsub, cudaStream_t s) {
  for (int i = 0; i < nsub; ++i) {
    const XeLaunch& L = subs[i];
    const int n = L.g.N * L.g.P;
    cudaError_t e = cudaMemsetAsync(L.counters, 0, 2 * sizeof(unsigned) * L.ring_slots, s);
    if (e == cudaSuccess && L.in_dtype == 0) {
      const size_t nseg = (L.g.Tp / kBK + std::max(1, L.ring_seg_kb) - 1) / std::max(1, L.ring_seg_kb);
      e = cudaMemsetAsync(L.amax, 0, sizeof(unsigned) * L.g.F * nseg, s);
    }
    if (e != cudaSuccess) return e;
    if (L.in_dtype != 0 && L.in_amax) {
      e = cudaMemsetAsync(L.in_amax, 0, sizeof(unsigned) * L.g.F * static_cast<size_t>(n), s);
      if (e != cudaSuccess) return e;
      // (The input is 16-byte aligned, so its rows are when they are a
      // multiple of 16 bytes.)
      if (L.in_dtype == 1)
        e = n % 4 == 0 ? launch_amax<1, 4>(L, n, s) : launch_amax<1, 1>(L, n, s);
      else
        e = n % 2 == 0 ? launch_amax<2, 2>(L, n, s) : launch_amax<2, 1>(L, n, s);
      if (e != cudaSuccess) return e;
    }
  }
  return cudaSuccess;
}

cudaError_t planar_launch(PlanarKernel& k, cudaStream_t s) {
  if (k.grid <= 0) return cudaSuccess;
  void* args[1] = {k.args};
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(static_cast<unsigned>(k.grid));
  cfg.blockDim = dim3(static_cast<unsigned>(k.block));
  cfg.dynamicSmemBytes = static_cast<size_t>(k.smem);
  cfg.stream = s;
  // The persistent CTAs wait on each other through the operand ring, so all
  // of them must be resident at once.  A cooperative launch guarantees that
  // or fails up front (cudaErrorCooperativeLaunchTooLarge, e.g. when part of
  // the GPU's SMs are held by another context), instead of a kernel whose
  // waits run out.  CTA-pair kernels rely on the cluster occupancy query of
  // planar_prepare instead.
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = k.shape == kShapePair ? 0 : 1;
  return cudaLaunchKernelExC(&cfg, k.func, args);
}

cudaError_t launch_planar(const CUtensorMap* in_map, const XeLaunch& L, int shape, cudaStream_t s) {
  static thread_local PlanarKernel k;
  const CUtensorMap* maps[1] = {in_map};
  cudaError_t e = planar_prepare(&L, maps, 1, &k, shape);
  if (e == cudaSuccess && k.grid > 0) e = planar_setup(&L, 1, s);
  if (e == cudaSuccess) e = planar_launch(k, s);
  return e;
}

}  // namespace xc
