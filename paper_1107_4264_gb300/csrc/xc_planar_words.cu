// xc_planar_words.cu -- the planar tensor-core X-engine's kernels for 8-bit rows
// that TMA cannot stride (xc_planar_kernel.cuh, converter_words), every tile
// shape, compiled apart from the others so they build in parallel.
#include "xc_planar_kernel.cuh"

namespace xc {

namespace {

template <int FMT, bool MULTI>
const void* words_kernel_of(int shape) {
  switch (shape) {
    case kShape128: return reinterpret_cast<const void*>(planar_kernel<true, 0, FMT, MULTI, kInWords>);
    case kShapePair: return reinterpret_cast<const void*>(planar_pair_kernel<true, 0, FMT, MULTI, kInWords>);
    case kShapeWide: return reinterpret_cast<const void*>(planar_wide_kernel<true, 0, FMT, MULTI, kInWords>);
    default: return nullptr;
  }
}

}  // namespace

const void* planar_words_select(int shape, int fmt, bool multi) {
  if (fmt == kFmtF8) return multi ? nullptr : words_kernel_of<kFmtF8, false>(shape);
  return multi ? words_kernel_of<kFmtF16, true>(shape) : words_kernel_of<kFmtF16, false>(shape);
}

}  // namespace xc
