// warp_bins.cuh -- the kernels of the warp and half-warp bins (H, W, W2) and
// their launchers, instantiated per precision in warp_bins_f32.cu and
// warp_bins_f64.cu (separate translation units compile in parallel).
#pragma once

#include "bin_queue.cuh"

namespace rsai {

template <typename T, int MODE>
__global__ void __launch_bounds__(256, (sizeof(T) == 8 ? 1 : 2))
    k_bin_warp(DevA A, DevParams P, Caps cap, ColQueue Q, ColOut O, Frozen F, unsigned long long *gctr, int last_bin) {
    extern __shared__ __align__(16) char smem[];
    const int wid = threadIdx.x >> 5;
    Work<T> w;
    w.carve(smem + (size_t)wid * Work<T>::bytes(cap), cap);
    WarpTeam team;
    run_queue<MODE>(team, w, A, P, cap, Q, O, F, gctr, last_bin != 0, 0);
}

// Bin H: every half warp is a team with its own workspace and its own column
template <typename T, int MODE>
__global__ void __launch_bounds__(256, (sizeof(T) == 8 ? 1 : 2))
    k_bin_half(DevA A, DevParams P, Caps cap, ColQueue Q, ColOut O, Frozen F, unsigned long long *gctr, int last_bin) {
    extern __shared__ __align__(16) char smem[];
    const int tid = threadIdx.x >> 4;
    Work<T> w;
    w.carve(smem + (size_t)tid * Work<T>::bytes(cap), cap);
    HalfTeam team;
    run_queue<MODE>(team, w, A, P, cap, Q, O, F, gctr, last_bin != 0, kBinHalf);
}

// ---------------------------------------------------------------------------
// host-side launchers

template <typename T, int MODE>
static cudaError_t launch_warp_m(int grid, int warps, const DevA &A, const DevParams &P, const Caps &cap,
                                 const ColQueue &Q, const ColOut &O, const Frozen &F, unsigned long long *gctr,
                                 bool last, cudaStream_t st) {
    const size_t smem = (size_t)warps * Work<T>::bytes(cap);
    allow_full_smem(k_bin_warp<T, MODE>);
    k_bin_warp<T, MODE><<<grid, warps * 32, smem, st>>>(A, P, cap, Q, O, F, gctr, last ? 1 : 0);
    return cudaGetLastError();
}

template <typename T, int MODE>
static cudaError_t launch_half_m(int grid, int warps, const DevA &A, const DevParams &P, const Caps &cap,
                                 const ColQueue &Q, const ColOut &O, const Frozen &F, unsigned long long *gctr,
                                 bool last, cudaStream_t st) {
    const size_t smem = (size_t)(2 * warps) * Work<T>::bytes(cap);
    allow_full_smem(k_bin_half<T, MODE>);
    k_bin_half<T, MODE><<<grid, warps * 32, smem, st>>>(A, P, cap, Q, O, F, gctr, last ? 1 : 0);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_warp_t(int mode, int grid, int warps, const DevA &A, const DevParams &P, const Caps &cap,
                            const ColQueue &Q, const ColOut &O, const Frozen &F, unsigned long long *gctr, bool last,
                            cudaStream_t st) {
    if (mode == MODE_BUILD) return launch_warp_m<T, MODE_BUILD>(grid, warps, A, P, cap, Q, O, F, gctr, last, st);
    if (mode == MODE_REFIT) return launch_warp_m<T, MODE_REFIT>(grid, warps, A, P, cap, Q, O, F, gctr, last, st);
    return launch_warp_m<T, MODE_BACKWARD>(grid, warps, A, P, cap, Q, O, F, gctr, last, st);
}

template <typename T>
cudaError_t launch_half_t(int mode, int grid, int warps, const DevA &A, const DevParams &P, const Caps &cap,
                            const ColQueue &Q, const ColOut &O, const Frozen &F, unsigned long long *gctr, bool last,
                            cudaStream_t st) {
    if (mode == MODE_BUILD) return launch_half_m<T, MODE_BUILD>(grid, warps, A, P, cap, Q, O, F, gctr, last, st);
    if (mode == MODE_REFIT) return launch_half_m<T, MODE_REFIT>(grid, warps, A, P, cap, Q, O, F, gctr, last, st);
    return launch_half_m<T, MODE_BACKWARD>(grid, warps, A, P, cap, Q, O, F, gctr, last, st);
}

template <typename T> int occupancy_warp_t(int warps, const Caps &cap) {
    int nb = 0;
    allow_full_smem(k_bin_warp<T, MODE_BUILD>);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_bin_warp<T, MODE_BUILD>, warps * 32,
                                                  (size_t)warps * Work<T>::bytes(cap));
    return nb;
}

template <typename T> int occupancy_half_t(int warps, const Caps &cap) {
    int nb = 0;
    allow_full_smem(k_bin_half<T, MODE_BUILD>);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_bin_half<T, MODE_BUILD>, warps * 32,
                                                  (size_t)(2 * warps) * Work<T>::bytes(cap));
    return nb;
}

#define RSAI_INSTANTIATE_WARP_BINS(T)                                                                               \
    template cudaError_t launch_warp_t<T>(int, int, int, const DevA &, const DevParams &, const Caps &,             \
                                          const ColQueue &, const ColOut &, const Frozen &, unsigned long long *,   \
                                          bool, cudaStream_t);                                                      \
    template cudaError_t launch_half_t<T>(int, int, int, const DevA &, const DevParams &, const Caps &,             \
                                          const ColQueue &, const ColOut &, const Frozen &, unsigned long long *,   \
                                          bool, cudaStream_t);                                                      \
    template int occupancy_warp_t<T>(int, const Caps &);                                                            \
    template int occupancy_half_t<T>(int, const Caps &);

}  // namespace rsai
