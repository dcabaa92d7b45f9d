// cta_build_f64.cu -- the CTA bins' build in FP64
#include "cta_bins.cuh"

namespace rsai {
RSAI_INSTANTIATE_CTA_MODE(double, MODE_BUILD)
RSAI_INSTANTIATE_CTA_OCCUPANCY(double)
}  // namespace rsai
