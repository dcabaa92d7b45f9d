// cta_bins.cuh -- the kernel of the CTA bins (S, C, G) and its launcher,
// instantiated per precision in cta_bins_f32.cu and cta_bins_f64.cu.
#pragma once

#include "bin_queue.cuh"

namespace rsai {

// NT threads per column.  STAGED: the workspace is a global-memory slab per CTA
// (gwork) and shared memory stages the panels; else it is in shared memory.
// MINB: CTAs per SM that the register budget has to allow.
template <typename T, int NT, bool STAGED, int MINB, int MODE>
__global__ void __launch_bounds__(NT, MINB)
    k_bin_block(DevA A, DevParams P, Caps cap, ColQueue Q, ColOut O, Frozen F, unsigned long long *gctr,
                int last_bin, char *gwork, size_t gstride, int bin, void *help, int owners) {
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

template <typename T, int NT, bool STAGED, int MINB, int MODE>
static cudaError_t launch_block_k(int grid, const DevA &A, const DevParams &P, const Caps &cap, const ColQueue &Q,
                                  const ColOut &O, const Frozen &F, unsigned long long *gctr, bool last, char *gwork,
                                  size_t gstride, int bin, void *help, int owners, cudaStream_t st) {
    const size_t smem = STAGED ? (size_t)cap.stage_bytes : Work<T>::bytes(cap);
    allow_full_smem(k_bin_block<T, NT, STAGED, MINB, MODE>);
    k_bin_block<T, NT, STAGED, MINB, MODE><<<grid, NT, smem, st>>>(A, P, cap, Q, O, F, gctr, last ? 1 : 0, gwork,
                                                                  gstride, bin, help, owners);
    return cudaGetLastError();
}

template <typename T, int MODE>
static cudaError_t launch_block_m(int kind, int grid, const DevA &A, const DevParams &P, const Caps &cap,
                                  const ColQueue &Q, const ColOut &O, const Frozen &F, unsigned long long *gctr,
                                  bool last, char *gwork, size_t gstride, int bin, void *help, int owners,
                                  cudaStream_t st) {
    if (kind == CTA_BIN_SMALL)
        return launch_block_k<T, kSmallThreads, false, kSmallCtas<T>, MODE>(grid, A, P, cap, Q, O, F, gctr, last,
                                                                            nullptr, 0, bin, nullptr, 0, st);
    if (kind == CTA_BIN_SHARED)
        return launch_block_k<T, kBlockThreads, false, 1, MODE>(grid, A, P, cap, Q, O, F, gctr, last, nullptr, 0, bin,
                                                                nullptr, 0, st);
    return launch_block_k<T, kBlockThreads, true, 1, MODE>(grid, A, P, cap, Q, O, F, gctr, last, gwork, gstride, bin,
                                                           help, owners, st);
}

template <typename T>
cudaError_t launch_block_t(int mode, int kind, int grid, const DevA &A, const DevParams &P, const Caps &cap,
                           const ColQueue &Q, const ColOut &O, const Frozen &F, unsigned long long *gctr, bool last,
                           char *gwork, size_t gstride, int bin, void *help, int owners, cudaStream_t st) {
    if (mode == MODE_BUILD)
        return launch_block_m<T, MODE_BUILD>(kind, grid, A, P, cap, Q, O, F, gctr, last, gwork, gstride, bin, help, owners,
                                             st);
    if (mode == MODE_REFIT)
        return launch_block_m<T, MODE_REFIT>(kind, grid, A, P, cap, Q, O, F, gctr, last, gwork, gstride, bin, help, owners,
                                             st);
    return launch_block_m<T, MODE_BACKWARD>(kind, grid, A, P, cap, Q, O, F, gctr, last, gwork, gstride, bin, help,
                                            owners, st);
}

// CTAs per SM of a bin with its workspace in shared memory
template <typename T> int occupancy_block_t(int kind, const Caps &cap) {
    int nb = 0;
    const size_t smem = Work<T>::bytes(cap);
    if (kind == CTA_BIN_SMALL) {
        allow_full_smem(k_bin_block<T, kSmallThreads, false, kSmallCtas<T>, MODE_BUILD>);
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(
            &nb, k_bin_block<T, kSmallThreads, false, kSmallCtas<T>, MODE_BUILD>, kSmallThreads, smem);
    } else {
        allow_full_smem(k_bin_block<T, kBlockThreads, false, 1, MODE_BUILD>);
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_bin_block<T, kBlockThreads, false, 1, MODE_BUILD>,
                                                      kBlockThreads, smem);
    }
    return nb;
}

#define RSAI_INSTANTIATE_CTA_BINS(T)                                                                                \
    template cudaError_t launch_block_t<T>(int, int, int, const DevA &, const DevParams &, const Caps &,            \
                                           const ColQueue &, const ColOut &, const Frozen &, unsigned long long *,  \
                                           bool, char *, size_t, int, void *, int, cudaStream_t);                   \
    template int occupancy_block_t<T>(int, const Caps &);

}  // namespace rsai
