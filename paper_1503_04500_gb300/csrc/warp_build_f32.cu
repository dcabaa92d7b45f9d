// warp_build_f32.cu -- the warp bins' build in FP32 (with FP64 refinement)
#include "warp_bins.cuh"

namespace rsai {
RSAI_INSTANTIATE_WARP_MODE(float, MODE_BUILD)
RSAI_INSTANTIATE_WARP_OCCUPANCY(float)
}  // namespace rsai
