// step_e4m3b.cu -- instantiations of the fused step kernel for E4M3 weights
// with FP16 block scales (one per 32 elements).
#include "step_kernel.cuh"

namespace mpadam {

template <int GD, int MD, bool SR, bool MIS>
static const void* pick_e4m3b(int options) {
  return options ? reinterpret_cast<const void*>(&step_kernel<kE4M3B, GD, MD, SR, true, MIS>)
                 : reinterpret_cast<const void*>(&step_kernel<kE4M3B, GD, MD, SR, false, MIS>);
}

template <int GD, int MD, bool MIS>
static const void* pick_e4m3b(int sr, int options) {
  return sr ? pick_e4m3b<GD, MD, true, MIS>(options) : pick_e4m3b<GD, MD, false, MIS>(options);
}

template <bool MIS>
static const void* pick_e4m3b_formats(int gd, int md, int sr, int options) {
  if (gd == kF32 && md == kF32) return pick_e4m3b<kF32, kF32, MIS>(sr, options);
  if (gd == kF32 && md == kBF16) return pick_e4m3b<kF32, kBF16, MIS>(sr, options);
  if (gd == kBF16 && md == kF32) return pick_e4m3b<kBF16, kF32, MIS>(sr, options);
  if (gd == kBF16 && md == kBF16) return pick_e4m3b<kBF16, kBF16, MIS>(sr, options);
  return nullptr;
}

const void* step_kernel_e4m3b(int gd, int md, int sr, int options, bool mis) {
  return mis ? pick_e4m3b_formats<true>(gd, md, sr, options) : pick_e4m3b_formats<false>(gd, md, sr, options);
}

}  // namespace mpadam
