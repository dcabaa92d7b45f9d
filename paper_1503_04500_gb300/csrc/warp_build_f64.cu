// warp_build_f64.cu -- the warp bins' build in FP64
#include "warp_bins.cuh"

namespace rsai {
RSAI_INSTANTIATE_WARP_MODE(double, MODE_BUILD)
RSAI_INSTANTIATE_WARP_OCCUPANCY(double)
}  // namespace rsai
