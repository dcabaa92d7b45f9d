// bin_queue.cuh -- the persistent loop of every size bin: columns pulled from an
// atomic queue, finished ones emitted to the result pool, ones that outgrow the
// bin forwarded to a larger bin's queue.  Shared by the warp bins
// (warp_bins.cuh) and the CTA bins (cta_bins.cuh).
#pragma once

#include "kernels.h"

namespace rsai {

// Column k to a larger bin's queue: the next bin or, where it is known to need
// |J| = need (0: not known) above wide_from, the first one that takes it.
__device__ __forceinline__ void forward_column(const ColQueue &Q, const ColOut &O, int32_t k, int need) {
    int32_t *cols = Q.ovf_cols;
    uint32_t *count = Q.ovf_count;
    if (Q.wide[0].cols != nullptr && need > Q.wide_from) {
        const int w = need <= Q.wide[0].pcap ? 0 : need <= Q.wide[1].pcap ? 1 : 2;
        cols = Q.wide[w].cols;
        count = Q.wide[w].count;
    }
    const uint32_t pos = atomicAdd(count, 1u);
    if ((int64_t)pos < Q.ovf_cap) cols[pos] = k;
    else set_error(O.err, RSAI_ERR_WORKSPACE);
}

template <class Team, typename T, class CapT>
__device__ void emit_or_forward(const Team &team, Column<Team, T, CapT> &col, int st, const ColQueue &Q,
                                const ColOut &O, bool last_bin, int bin) {
    const int me = team.rank();
    const int32_t k = col.k;
    Work<T> &w = col.w;
    if (st != COL_DONE) {
        if (!last_bin) {
            if (me == 0) forward_column(Q, O, k, st == COL_OVERFLOW_J ? col.need : 0);
        } else if (me == 0) {
            O.col_off[k] = 0;
            O.col_len[k] = 0;
            O.col_q[k] = 0;
            O.rho[k] = NAN;
            O.loops[k] = 0;
            O.flags[k] = RSAI_COL_FAILED;
            w.ctr[CTR_FAILED] += 1;
            set_error(O.err, RSAI_ERR_WORKSPACE);
        }
        team.sync();
        return;
    }
    const int p = col.p;
    unsigned long long off = 0;
    if (me == 0) off = atomicAdd(O.pool_top, (unsigned long long)p);
    off = team.bcast(off, 0);
    if ((int64_t)(off + p) > O.pool_cap) {
        if (me == 0) {
            O.col_off[k] = 0;
            O.col_len[k] = 0;
            O.col_q[k] = 0;
            O.rho[k] = NAN;
            O.loops[k] = 0;
            O.flags[k] = RSAI_COL_FAILED;
            w.ctr[CTR_FAILED] += 1;
            set_error(O.err, RSAI_ERR_WORKSPACE);
        }
        team.sync();
        return;
    }
    int fin = 1;
    for (int c = me; c < p; c += Team::SIZE) {
        O.pool_rows[off + c] = w.J[c];
        O.pool_vals[off + c] = w.m[c];
        fin &= finite_bits(w.m[c]) ? 1 : 0;
    }
    fin = team.sum(1 - fin) == 0 && finite_bits(col.rho);
    if (me == 0) {
        int flags = (col.rho <= col.P.eps ? RSAI_COL_CONVERGED : 0) | (col.rank_flag ? RSAI_COL_RANK : 0) |
                    (fin ? 0 : RSAI_COL_NONFINITE);
        O.col_off[k] = (int64_t)off;
        O.col_len[k] = p;
        O.col_q[k] = col.q;
        O.rho[k] = col.rho;
        O.loops[k] = col.l;
        O.flags[k] = flags;
        w.ctr[CTR_QR] += col.c_qr;
        w.ctr[CTR_RES] += col.c_res;
        w.ctr[CTR_REFINE] += col.c_ref;
        w.ctr[CTR_REFINE64] += col.c_ref64;
        w.ctr[CTR_BYTES] += col.c_bytes;
        w.ctr[CTR_SELECT] += col.c_sel;
        w.ctr[CTR_LOOPS] += col.l;
        w.ctr[CTR_SOLVES] += col.c_solves;
        w.ctr[CTR_DROPS] += col.c_drops;
        w.ctr[CTR_PMAX] = max(w.ctr[CTR_PMAX], (long long)col.c_pmax);
        w.ctr[CTR_QMAX] = max(w.ctr[CTR_QMAX], (long long)col.c_qmax);
        w.ctr[CTR_COLS] += 1;
        w.ctr[CTR_RANK] += col.rank_flag ? 1 : 0;
        w.ctr[CTR_NONFINITE] += fin ? 0 : 1;
    }
    team.sync();
    (void)bin;
}

// A frozen-pattern column that does not fit this bin: forward or fail
__device__ __forceinline__ void forward_frozen(int me, const ColQueue &Q, const ColOut &O, int32_t k,
                                               bool last_bin, int need, long long *ctr) {
    if (me != 0) return;
    if (!last_bin) {
        forward_column(Q, O, k, need);
    } else {
        ctr[CTR_FAILED] += 1;
        set_error(O.err, RSAI_ERR_WORKSPACE);
    }
}

// A bin that no column was forwarded to (the counts are final when its kernel
// starts): its CTAs return before they set up anything.  The five or six empty
// bins of a stencil matrix took a twentieth of a small build (with the launches, copies
// and allocations saved elsewhere in a build: 20^2 in FP64 793 -> 692 us, rebuild of
// 256^2 1050 -> 1000 us, its refit and adjoint 1884 -> 1728 us).
__device__ __forceinline__ bool queue_empty(const ColQueue &Q) {
    return Q.count != nullptr && *(volatile const uint32_t *)Q.count == 0u;
}

template <int MODE, class Team, typename T, class CapT>
__device__ void run_queue(const Team &team, Work<T> &w, const DevA &A, const DevParams &P, const CapT &cap,
                          const ColQueue &Q, const ColOut &O, const Frozen &F, unsigned long long *gctr,
                          bool last_bin, int bin) {
    const int me = team.rank();
    for (int i = me; i < CTR_COUNT; i += Team::SIZE) w.ctr[i] = 0;
    team.sync();
    const int64_t nq = Q.count ? (int64_t)(*(volatile const uint32_t *)Q.count) : Q.n;
    // Half-warp teams: the two halves of a warp start their columns together
    // (one vote of the whole warp per column), so that similar columns run in
    // step and each instruction serves both; a half whose queue is empty sits
    // the round out.  The loop ends only when neither half has a column, so
    // every lane of the warp reaches each whole-warp vote and synchronisation.
    constexpr bool paired = std::is_same<Team, HalfTeam>::value;
    for (;;) {
        uint32_t idx = 0;
        if (me == 0) idx = atomicAdd(Q.next, 1u);
        idx = team.bcast(idx, 0);
        const bool have = (int64_t)idx < nq;
        if constexpr (paired) {
            if (!__any_sync(0xffffffffu, have)) break;
        } else {
            if (!have) break;
        }
        if (have) {
            const int32_t k = Q.cols ? Q.cols[idx] : (int32_t)idx;
            Column<Team, T, CapT> col(team, A, P, cap, w, k);
            if constexpr (MODE == MODE_BUILD) {
                int st = col.run();
                emit_or_forward(team, col, st, Q, O, last_bin, bin);
            } else {
                const int64_t mo = F.Mcolptr[k];
                const int pk = (int)(F.Mcolptr[k + 1] - mo);
                bool ok = col.load_pattern(F.Mrows + mo, pk);
                if (ok) {
                    if constexpr (MODE == MODE_REFIT) ok = col.refit();
                    else ok = col.adjoint(F);
                }
                if (!ok) {
                    forward_frozen(me, Q, O, k, last_bin, pk > cap.pcap ? pk : 0, w.ctr);
                } else {
                    if constexpr (MODE == MODE_REFIT) {
                        for (int c = me; c < pk; c += Team::SIZE) F.Mval_csr[F.Mcsc_to_csr[mo + c]] = w.m[c];
                        if (me == 0) F.rho2[k] = col.rho * col.rho;
                    }
                    if (me == 0) w.ctr[CTR_COLS] += 1;
                }
                team.sync();
            }
        }
        if constexpr (paired) __syncwarp();
        if constexpr (Team::STAGED) {
            if (have && me == 0) atomicAdd(w.ho->board.cols_done, 1u);
        }
    }
    team.sync();
    if (me == 0) {
        for (int i = 0; i < CTR_COUNT; ++i) {
            if (i == CTR_PMAX || i == CTR_QMAX)
                atomicMax(&gctr[i], (unsigned long long)w.ctr[i]);
            else if (w.ctr[i] != 0)
                atomicAdd(&gctr[i], (unsigned long long)w.ctr[i]);
        }
        if (w.ctr[CTR_COLS] != 0) atomicAdd(&gctr[CTR_COUNT + bin], (unsigned long long)w.ctr[CTR_COLS]);
    }
}

// ---------------------------------------------------------------------------
// host side

// Lets `fn` take up to the device's opt-in shared memory per block, less its
// static shared memory.  The limit is raised to that largest value instead of
// to each launch's size, so that every launch recorded in a CUDA graph stays
// within the function's limit whatever was launched (or planned) after it.
template <typename F> static void allow_full_smem(F fn) {
    int dev = 0, optin = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    cudaFuncAttributes fa{};
    cudaFuncGetAttributes(&fa, fn);  // static + dynamic must not exceed the opt-in limit
    cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, optin - (int)fa.sharedSizeBytes);
}

}  // namespace rsai
