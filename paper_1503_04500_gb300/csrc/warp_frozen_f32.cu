// warp_frozen_f32.cu -- the warp bins' frozen-pattern passes in FP32 (with FP64 refinement)
#include "warp_bins.cuh"

namespace rsai {
RSAI_INSTANTIATE_WARP_MODE(float, MODE_REFIT)
RSAI_INSTANTIATE_WARP_MODE(float, MODE_BACKWARD)
}  // namespace rsai
