// cta_bins_f64.cu -- the CTA bins in FP64
#include "cta_bins.cuh"

namespace rsai {
RSAI_INSTANTIATE_CTA_BINS(double)
}  // namespace rsai
