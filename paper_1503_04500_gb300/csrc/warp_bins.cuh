// warp_bins.cuh -- the kernels of the warp and half-warp bins (H, W0, W, W2) and
// their launchers, instantiated per precision and mode in warp_build_*.cu and
// warp_frozen_*.cu (separate translation units compile in parallel).
#pragma once

#include "bin_queue.cuh"

namespace rsai {

// The sizes of the warp bins (plan_bins fills the same numbers into Caps)
using CapsW0 = FixedCaps<48, 16, 128, 32, 32>;
using CapsW = FixedCaps<64, 32, 256, 64, 64>;
using CapsW2 = FixedCaps<128, 32, 512, 64, 128>;
using CapsH = CapsW0;

// CTAs per SM that the register budget of 256 threads has to allow
template <typename T, class CapT> constexpr int kWarpCtas = sizeof(T) == 8 ? 1 : CapT::qcap <= 48 ? 3 : 2;
template <typename T> constexpr int kWarpCtas<T, Caps> = sizeof(T) == 8 ? 1 : 2;

template <typename T, int MODE, class CapT>
__global__ void __launch_bounds__(256, kWarpCtas<T, CapT>)
    k_bin_warp(DevA A, DevParams P, CapT cap, ColQueue Q, ColOut O, Frozen F, unsigned long long *gctr, int last_bin) {
    if (queue_empty(Q)) return;
    extern __shared__ __align__(16) char smem[];
    const int wid = threadIdx.x >> 5;
    Work<T> w;
    w.carve(smem + (size_t)wid * Work<T>::bytes(cap), cap);
    WarpTeam team;
    run_queue<MODE>(team, w, A, P, cap, Q, O, F, gctr, last_bin != 0, 0);
}

// Bin H: every half warp is a team with its own workspace and its own column
template <typename T, int MODE, class CapT>
__global__ void __launch_bounds__(256, (sizeof(T) == 8 ? 1 : 2))
    k_bin_half(DevA A, DevParams P, CapT cap, ColQueue Q, ColOut O, Frozen F, unsigned long long *gctr, int last_bin) {
    if (queue_empty(Q)) return;
    extern __shared__ __align__(16) char smem[];
    const int tid = threadIdx.x >> 4;
    Work<T> w;
    w.carve(smem + (size_t)tid * Work<T>::bytes(cap), cap);
    HalfTeam team;
    run_queue<MODE>(team, w, A, P, cap, Q, O, F, gctr, last_bin != 0, kBinHalf);
}

// ---------------------------------------------------------------------------
// host-side launchers

template <typename T, int MODE, class CapT>
static cudaError_t launch_warp_c(int grid, int warps, const DevA &A, const DevParams &P, const CapT &cap,
                                 const ColQueue &Q, const ColOut &O, const Frozen &F, unsigned long long *gctr,
                                 bool last, cudaStream_t st) {
    allow_full_smem(k_bin_warp<T, MODE, CapT>);
    k_bin_warp<T, MODE, CapT><<<grid, warps * 32, (size_t)warps * Work<T>::bytes(cap), st>>>(A, P, cap, Q, O, F, gctr,
                                                                                            last ? 1 : 0);
    return cudaGetLastError();
}

template <typename T, int MODE>
cudaError_t launch_warp_m(int grid, int warps, const DevA &A, const DevParams &P, const Caps &cap,
                                 const ColQueue &Q, const ColOut &O, const Frozen &F, unsigned long long *gctr,
                                 bool last, cudaStream_t st) {
    constexpr bool build = MODE == MODE_BUILD;
    if (build ? CapsW0::fits(cap) : CapsW0::fits_frozen(cap))
        return launch_warp_c<T, MODE>(grid, warps, A, P, CapsW0{cap.small_p}, Q, O, F, gctr, last, st);
    if (build ? CapsW::fits(cap) : CapsW::fits_frozen(cap))
        return launch_warp_c<T, MODE>(grid, warps, A, P, CapsW{cap.small_p}, Q, O, F, gctr, last, st);
    if (build ? CapsW2::fits(cap) : CapsW2::fits_frozen(cap))
        return launch_warp_c<T, MODE>(grid, warps, A, P, CapsW2{cap.small_p}, Q, O, F, gctr, last, st);
    if constexpr (build) return launch_warp_c<T, MODE>(grid, warps, A, P, cap, Q, O, F, gctr, last, st);
    else return cudaErrorInvalidValue;
}

template <typename T, int MODE, class CapT>
static cudaError_t launch_half_c(int grid, int warps, const DevA &A, const DevParams &P, const CapT &cap,
                                 const ColQueue &Q, const ColOut &O, const Frozen &F, unsigned long long *gctr,
                                 bool last, cudaStream_t st) {
    allow_full_smem(k_bin_half<T, MODE, CapT>);
    k_bin_half<T, MODE, CapT><<<grid, warps * 32, (size_t)(2 * warps) * Work<T>::bytes(cap), st>>>(
        A, P, cap, Q, O, F, gctr, last ? 1 : 0);
    return cudaGetLastError();
}

template <typename T, int MODE>
cudaError_t launch_half_m(int grid, int warps, const DevA &A, const DevParams &P, const Caps &cap,
                                 const ColQueue &Q, const ColOut &O, const Frozen &F, unsigned long long *gctr,
                                 bool last, cudaStream_t st) {
    if (MODE == MODE_BUILD ? CapsH::fits(cap) : CapsH::fits_frozen(cap))
        return launch_half_c<T, MODE>(grid, warps, A, P, CapsH{cap.small_p}, Q, O, F, gctr, last, st);
    if constexpr (MODE == MODE_BUILD) return launch_half_c<T, MODE>(grid, warps, A, P, cap, Q, O, F, gctr, last, st);
    else return cudaErrorInvalidValue;
}

template <typename T, class CapT> static int occupancy_warp_c(int warps, const CapT &cap) {
    int nb = 0;
    allow_full_smem(k_bin_warp<T, MODE_BUILD, CapT>);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_bin_warp<T, MODE_BUILD, CapT>, warps * 32,
                                                  (size_t)warps * Work<T>::bytes(cap));
    return nb;
}

template <typename T> int occupancy_warp_t(int warps, const Caps &cap) {
    if (CapsW0::fits(cap)) return occupancy_warp_c<T>(warps, CapsW0{cap.small_p});
    if (CapsW::fits(cap)) return occupancy_warp_c<T>(warps, CapsW{cap.small_p});
    if (CapsW2::fits(cap)) return occupancy_warp_c<T>(warps, CapsW2{cap.small_p});
    return occupancy_warp_c<T>(warps, cap);
}

template <typename T, class CapT> static int occupancy_half_c(int warps, const CapT &cap) {
    int nb = 0;
    allow_full_smem(k_bin_half<T, MODE_BUILD, CapT>);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_bin_half<T, MODE_BUILD, CapT>, warps * 32,
                                                  (size_t)(2 * warps) * Work<T>::bytes(cap));
    return nb;
}

template <typename T> int occupancy_half_t(int warps, const Caps &cap) {
    if (CapsH::fits(cap)) return occupancy_half_c<T>(warps, CapsH{cap.small_p});
    return occupancy_half_c<T>(warps, cap);
}

#define RSAI_INSTANTIATE_WARP_MODE(T, MODE)                                                                         \
    template cudaError_t launch_warp_m<T, MODE>(int, int, const DevA &, const DevParams &, const Caps &,            \
                                                const ColQueue &, const ColOut &, const Frozen &,                   \
                                                unsigned long long *, bool, cudaStream_t);                          \
    template cudaError_t launch_half_m<T, MODE>(int, int, const DevA &, const DevParams &, const Caps &,            \
                                                const ColQueue &, const ColOut &, const Frozen &,                   \
                                                unsigned long long *, bool, cudaStream_t);
#define RSAI_INSTANTIATE_WARP_OCCUPANCY(T)               \
    template int occupancy_warp_t<T>(int, const Caps &); \
    template int occupancy_half_t<T>(int, const Caps &);

}  // namespace rsai
