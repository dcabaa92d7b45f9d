// cta_bins.cuh -- the kernel of the CTA bins (S0, S, C, G) and its launcher,
// instantiated per precision and mode in cta_build_*.cu and cta_frozen_*.cu.
#pragma once

#include "bin_queue.cuh"

namespace rsai {

// The sizes of bins S0 and S (plan_bins fills the same numbers into Caps when c * l_max <= 64;
// above, R is larger and the layout is the runtime one: 200^2 at eps = 0.12, CTA bins in
// FP32 108.9 ms with c * l_max = 64, 112.8 with 66, in FP64 232 both)
using CapsS0 = FixedCaps<96, 40, 256, 64, 128, 1>;
using CapsS = FixedCaps<128, 64, 512, 64, 256, 1>;

// NT threads per column.  STAGED: the workspace is a global-memory slab per CTA
// (gwork) and shared memory stages the panels; else it is in shared memory.
// MINB: CTAs per SM that the register budget has to allow.
template <typename T, int NT, bool STAGED, int MINB, int MODE, class CapT>
__global__ void __launch_bounds__(NT, MINB)
    k_bin_block(DevA A, DevParams P, CapT cap, ColQueue Q, ColOut O, Frozen F, unsigned long long *gctr,
                int last_bin, char *gwork, size_t gstride, int bin, void *help, int owners) {
    if (queue_empty(Q)) return;
    extern __shared__ __align__(16) char smem[];
    __shared__ unsigned long long red[kVirtualWarps + 1];
    __shared__ int redi[kVirtualWarps + 1];
    BlockTeam<NT, STAGED> team{red, redi};
    if constexpr (STAGED) {
        // CTAs beyond the owners have no workspace: they only help
        __shared__ HelpOwner ho;
        if (threadIdx.x == 0) ho = HelpOwner{HelpBoard::at(help, owners), (int)blockIdx.x, 0u, O.err};
        __syncthreads();
        if ((int)blockIdx.x < owners) {
            Work<T> w;
            w.carve(gwork + (size_t)blockIdx.x * gstride, cap);
            w.stage = smem;  // shared memory is free for panel staging
            w.ho = &ho;
            run_queue<MODE>(team, w, A, P, cap, Q, O, F, gctr, last_bin != 0, bin);
        }
        help_others<BlockTeam<NT, STAGED>, T>(team, ho.board, *Q.count, (T *)smem);
    } else {
        Work<T> w;
        w.carve(smem, cap);
        run_queue<MODE>(team, w, A, P, cap, Q, O, F, gctr, last_bin != 0, bin);
    }
}

// ---------------------------------------------------------------------------
// host-side launchers

template <typename T, int NT, bool STAGED, int MINB, int MODE, class CapT>
static cudaError_t launch_block_k(int grid, const DevA &A, const DevParams &P, const CapT &cap, const ColQueue &Q,
                                  const ColOut &O, const Frozen &F, unsigned long long *gctr, bool last, char *gwork,
                                  size_t gstride, int bin, void *help, int owners, cudaStream_t st) {
    const size_t smem = STAGED ? (size_t)cap.stage_bytes : Work<T>::bytes(cap);
    allow_full_smem(k_bin_block<T, NT, STAGED, MINB, MODE, CapT>);
    k_bin_block<T, NT, STAGED, MINB, MODE, CapT><<<grid, NT, smem, st>>>(A, P, cap, Q, O, F, gctr, last ? 1 : 0, gwork,
                                                                  gstride, bin, help, owners);
    return cudaGetLastError();
}

template <typename T, int MODE>
cudaError_t launch_block_m(int kind, int grid, const DevA &A, const DevParams &P, const Caps &cap, const ColQueue &Q,
                           const ColOut &O, const Frozen &F, unsigned long long *gctr, bool last, char *gwork,
                           size_t gstride, int bin, void *help, int owners, cudaStream_t st) {
    constexpr bool build = MODE == MODE_BUILD;
    if (kind == CTA_BIN_TINY) {
        if (build ? CapsS0::fits(cap) : CapsS0::fits_frozen(cap))
            return launch_block_k<T, kTinyThreads, false, kTinyCtas<T>, MODE>(
                grid, A, P, CapsS0{0}, Q, O, F, gctr, last, nullptr, 0, bin, nullptr, 0, st);
        if constexpr (build)
            return launch_block_k<T, kTinyThreads, false, kTinyCtas<T>, MODE>(grid, A, P, cap, Q, O, F, gctr, last,
                                                                              nullptr, 0, bin, nullptr, 0, st);
        return cudaErrorInvalidValue;
    }
    if (kind == CTA_BIN_SMALL) {
        if (build ? CapsS::fits(cap) : CapsS::fits_frozen(cap))
            return launch_block_k<T, kSmallThreads, false, kSmallCtas<T>, MODE>(
                grid, A, P, CapsS{0}, Q, O, F, gctr, last, nullptr, 0, bin, nullptr, 0, st);
        if constexpr (build)
            return launch_block_k<T, kSmallThreads, false, kSmallCtas<T>, MODE>(grid, A, P, cap, Q, O, F, gctr, last,
                                                                                nullptr, 0, bin, nullptr, 0, st);
        return cudaErrorInvalidValue;
    }
    if (kind == CTA_BIN_SHARED)
        return launch_block_k<T, kBlockThreads, false, 1, MODE>(grid, A, P, cap, Q, O, F, gctr, last, nullptr, 0, bin,
                                                                nullptr, 0, st);
    return launch_block_k<T, kBlockThreads, true, 1, MODE>(grid, A, P, cap, Q, O, F, gctr, last, gwork, gstride, bin,
                                                           help, owners, st);
}

// CTAs per SM of a bin with its workspace in shared memory
template <typename T, int NT, int MINB, class CapT> static int occupancy_block_c(const CapT &cap) {
    int nb = 0;
    allow_full_smem(k_bin_block<T, NT, false, MINB, MODE_BUILD, CapT>);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_bin_block<T, NT, false, MINB, MODE_BUILD, CapT>, NT,
                                                  Work<T>::bytes(cap));
    return nb;
}

template <typename T> int occupancy_block_t(int kind, const Caps &cap) {
    if (kind == CTA_BIN_TINY && CapsS0::fits(cap)) return occupancy_block_c<T, kTinyThreads, kTinyCtas<T>>(CapsS0{0});
    if (kind == CTA_BIN_TINY) return occupancy_block_c<T, kTinyThreads, kTinyCtas<T>>(cap);
    if (kind == CTA_BIN_SMALL && CapsS::fits(cap)) return occupancy_block_c<T, kSmallThreads, kSmallCtas<T>>(CapsS{0});
    if (kind == CTA_BIN_SMALL) return occupancy_block_c<T, kSmallThreads, kSmallCtas<T>>(cap);
    return occupancy_block_c<T, kBlockThreads, 1>(cap);
}

#define RSAI_INSTANTIATE_CTA_MODE(T, MODE)                                                                          \
    template cudaError_t launch_block_m<T, MODE>(int, int, const DevA &, const DevParams &, const Caps &,           \
                                                 const ColQueue &, const ColOut &, const Frozen &,                  \
                                                 unsigned long long *, bool, char *, size_t, int, void *, int,      \
                                                 cudaStream_t);
#define RSAI_INSTANTIATE_CTA_OCCUPANCY(T) template int occupancy_block_t<T>(int, const Caps &);

}  // namespace rsai
