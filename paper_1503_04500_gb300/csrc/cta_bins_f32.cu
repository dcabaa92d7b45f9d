// cta_bins_f32.cu -- the CTA bins in FP32 (with FP64 refinement)
#include "cta_bins.cuh"

namespace rsai {
RSAI_INSTANTIATE_CTA_BINS(float)
}  // namespace rsai
