// cta_frozen_f32.cu -- the CTA bins' frozen-pattern passes in FP32 (with FP64 refinement)
#include "cta_bins.cuh"

namespace rsai {
RSAI_INSTANTIATE_CTA_MODE(float, MODE_REFIT)
RSAI_INSTANTIATE_CTA_MODE(float, MODE_BACKWARD)
}  // namespace rsai
