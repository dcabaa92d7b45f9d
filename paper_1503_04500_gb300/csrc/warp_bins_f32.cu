// warp_bins_f32.cu -- the warp bins in FP32 (with FP64 refinement)
#include "warp_bins.cuh"

namespace rsai {
RSAI_INSTANTIATE_WARP_BINS(float)
}  // namespace rsai
