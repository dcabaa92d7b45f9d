// warp_bins_f64.cu -- the warp bins in FP64
#include "warp_bins.cuh"

namespace rsai {
RSAI_INSTANTIATE_WARP_BINS(double)
}  // namespace rsai
