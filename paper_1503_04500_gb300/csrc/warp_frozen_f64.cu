// warp_frozen_f64.cu -- the warp bins' frozen-pattern passes in FP64
#include "warp_bins.cuh"

namespace rsai {
RSAI_INSTANTIATE_WARP_MODE(double, MODE_REFIT)
RSAI_INSTANTIATE_WARP_MODE(double, MODE_BACKWARD)
}  // namespace rsai
