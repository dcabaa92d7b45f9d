// cta_frozen_f64.cu -- the CTA bins' frozen-pattern passes in FP64
#include "cta_bins.cuh"

namespace rsai {
RSAI_INSTANTIATE_CTA_MODE(double, MODE_REFIT)
RSAI_INSTANTIATE_CTA_MODE(double, MODE_BACKWARD)
}  // namespace rsai
