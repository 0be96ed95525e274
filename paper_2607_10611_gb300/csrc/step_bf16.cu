// step_bf16.cu -- instantiations of the fused step kernel for BF16 weights.
#include "step_kernel.cuh"

namespace mpadam {

template <int GD, int MD, bool SR, bool MIS>
static const void* pick_bf16(int options) {
  return options ? reinterpret_cast<const void*>(&step_kernel<kBF16, GD, MD, SR, true, MIS>)
                 : reinterpret_cast<const void*>(&step_kernel<kBF16, GD, MD, SR, false, MIS>);
}

template <int GD, int MD, bool MIS>
static const void* pick_bf16(int sr, int options) {
  return sr ? pick_bf16<GD, MD, true, MIS>(options) : pick_bf16<GD, MD, false, MIS>(options);
}

template <bool MIS>
static const void* pick_bf16_formats(int gd, int md, int sr, int options) {
  if (gd == kF32 && md == kF32) return pick_bf16<kF32, kF32, MIS>(sr, options);
  if (gd == kF32 && md == kBF16) return pick_bf16<kF32, kBF16, MIS>(sr, options);
  if (gd == kBF16 && md == kF32) return pick_bf16<kBF16, kF32, MIS>(sr, options);
  if (gd == kBF16 && md == kBF16) return pick_bf16<kBF16, kBF16, MIS>(sr, options);
  return nullptr;
}

const void* step_kernel_bf16(int gd, int md, int sr, int options, bool mis) {
  return mis ? pick_bf16_formats<true>(gd, md, sr, options) : pick_bf16_formats<false>(gd, md, sr, options);
}

}  // namespace mpadam
