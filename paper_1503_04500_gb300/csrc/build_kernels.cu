// build_kernels.cu -- the size bins of the RSAI(tol) column algorithm and
// their launchers (input checks, ||A||_1, statistics and the assembly of M
// are in setup_kernels.cu).
//
// Bins (one persistent launch each, columns pulled from an atomic queue; the
// columns are independent, Section 2 Eq. 2.2):
//   H  half a warp per column, two columns per warp, workspace in shared
//      memory (|I| <= 48, |J| <= 16, e.g. 3-D 7-point stencils; first bin in FP64)
//   W0 one warp per column, the same sizes (first bin in FP32)
//   W  one warp per column (|I| <= 64, |J| <= 32)
//   W2 the same kernel with |I| <= 128 (fewer warps per SM)
//   S0 one CTA of 64 threads per column, workspace in shared memory (|I| <= 96, |J| <= 40)
//   S  one CTA of 128 threads (|I| <= 128, |J| <= 64)
//   C  one CTA per column, workspace in shared memory (up to ~200 KB)
//   G  one CTA per column, workspace in a global-memory slab per CTA (the
//      long tail of matrices with dense rows, Section 4 "row irregular")
// A column that outgrows a bin is pushed to the next bin's queue (past those too
// narrow for its |J|) and restarted there from J = {k}; the result is the same column of M.
#include "kernels.h"

namespace rsai {

// ---------------------------------------------------------------------------
// dispatch on the precision (the kernels are in warp_bins.cuh and cta_bins.cuh)

template <typename T>
size_t work_bytes(const Caps &c) { return Work<T>::bytes(c); }

template size_t work_bytes<float>(const Caps &);
template size_t work_bytes<double>(const Caps &);

template <typename T, typename... Args> static cudaError_t warp_by_mode(int mode, Args &&...a) {
    if (mode == MODE_BUILD) return launch_warp_m<T, MODE_BUILD>(a...);
    if (mode == MODE_REFIT) return launch_warp_m<T, MODE_REFIT>(a...);
    return launch_warp_m<T, MODE_BACKWARD>(a...);
}
template <typename T, typename... Args> static cudaError_t half_by_mode(int mode, Args &&...a) {
    if (mode == MODE_BUILD) return launch_half_m<T, MODE_BUILD>(a...);
    if (mode == MODE_REFIT) return launch_half_m<T, MODE_REFIT>(a...);
    return launch_half_m<T, MODE_BACKWARD>(a...);
}
template <typename T, typename... Args> static cudaError_t block_by_mode(int mode, Args &&...a) {
    if (mode == MODE_BUILD) return launch_block_m<T, MODE_BUILD>(a...);
    if (mode == MODE_REFIT) return launch_block_m<T, MODE_REFIT>(a...);
    return launch_block_m<T, MODE_BACKWARD>(a...);
}

cudaError_t launch_bin_warp(int mode, bool fp32, int grid, int warps, const DevA &A, const DevParams &P,
                            const Caps &cap, const ColQueue &Q, const ColOut &O, const Frozen &F,
                            unsigned long long *gctr, bool last, cudaStream_t st) {
    return fp32 ? warp_by_mode<float>(mode, grid, warps, A, P, cap, Q, O, F, gctr, last, st)
                : warp_by_mode<double>(mode, grid, warps, A, P, cap, Q, O, F, gctr, last, st);
}

cudaError_t launch_bin_half(int mode, bool fp32, int grid, int warps, const DevA &A, const DevParams &P,
                            const Caps &cap, const ColQueue &Q, const ColOut &O, const Frozen &F,
                            unsigned long long *gctr, bool last, cudaStream_t st) {
    return fp32 ? half_by_mode<float>(mode, grid, warps, A, P, cap, Q, O, F, gctr, last, st)
                : half_by_mode<double>(mode, grid, warps, A, P, cap, Q, O, F, gctr, last, st);
}

cudaError_t launch_bin_block(int mode, bool fp32, int kind, int grid, const DevA &A, const DevParams &P,
                             const Caps &cap, const ColQueue &Q, const ColOut &O, const Frozen &F,
                             unsigned long long *gctr, bool last, char *gwork, size_t gstride, int bin, void *help,
                             int owners, cudaStream_t st) {
    return fp32 ? block_by_mode<float>(mode, kind, grid, A, P, cap, Q, O, F, gctr, last, gwork, gstride, bin, help,
                                       owners, st)
                : block_by_mode<double>(mode, kind, grid, A, P, cap, Q, O, F, gctr, last, gwork, gstride, bin, help,
                                        owners, st);
}

int occupancy_bin_warp(bool fp32, int warps, const Caps &cap) {
    return fp32 ? occupancy_warp_t<float>(warps, cap) : occupancy_warp_t<double>(warps, cap);
}

int occupancy_bin_half(bool fp32, int warps, const Caps &cap) {
    return fp32 ? occupancy_half_t<float>(warps, cap) : occupancy_half_t<double>(warps, cap);
}

int occupancy_bin_block(bool fp32, int kind, const Caps &cap) {
    return fp32 ? occupancy_block_t<float>(kind, cap) : occupancy_block_t<double>(kind, cap);
}

}  // namespace rsai
