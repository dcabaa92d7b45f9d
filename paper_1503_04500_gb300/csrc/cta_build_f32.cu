// cta_build_f32.cu -- the CTA bins' build in FP32 (with FP64 refinement)
#include "cta_bins.cuh"

namespace rsai {
RSAI_INSTANTIATE_CTA_MODE(float, MODE_BUILD)
RSAI_INSTANTIATE_CTA_OCCUPANCY(float)
}  // namespace rsai
