// spmv.cuh -- rows of a CSR product, shared by rsai_spmv / rsai_apply and the solver
#pragma once

#include <stdint.h>

namespace rsai {

struct CsrView {
    const int64_t *row_ptr;
    const int32_t *col_idx;
    const double *val;
};

// Rows that a group of 8 lanes takes at a time
constexpr int kRowsPerGroup = 4;

// y[row0 .. row0 + 4) = (A x) of these rows (rows >= end: nothing), on the 8
// lanes sub = 0..7 of a group; every lane of the warp calls.  Lane sub of a row
// adds entries sub, sub + 8, ... in order and a butterfly over 4, 2, 1 joins the
// lanes.  Four rows at a time: their loads are in flight together, and the
// butterflies are one reduce-scatter (4 additions per lane for four rows
// instead of 12, the same sums): on this GPU's FP64 unit (2 lanes per cycle and
// SM) the additions of one butterfly per row took longer than the products of
// a row of 16 entries.
__device__ __forceinline__ void spmv_rows(const CsrView &A, const double *x, double *y, int64_t row0, int64_t end,
                                          int sub) {
    static_assert(kRowsPerGroup == 4, "the exchange below is written for four rows");
    int64_t at[4];
    int len[4];
    int most = 0;
    int64_t a = row0 < end ? A.row_ptr[row0] : 0;
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        const int64_t b = row0 + r < end ? A.row_ptr[row0 + r + 1] : a;
        at[r] = a;
        len[r] = (int)(b - a);
        most = max(most, len[r]);
        a = b;
    }
    double acc[4] = {0.0, 0.0, 0.0, 0.0};
    for (int e = sub; e < most; e += 8) {
        int32_t c[4];
        double v[4];
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            c[r] = e < len[r] ? A.col_idx[at[r] + e] : -1;
            v[r] = e < len[r] ? A.val[at[r] + e] : 0.0;
        }
#pragma unroll
        for (int r = 0; r < 4; ++r)
            if (c[r] >= 0) acc[r] = fma(v[r], x[c[r]], acc[r]);
    }
    const bool hi = sub & 4, mid = sub & 2;
    const double s0 = (hi ? acc[2] : acc[0]) + __shfl_xor_sync(0xffffffffu, hi ? acc[0] : acc[2], 4);
    const double s1 = (hi ? acc[3] : acc[1]) + __shfl_xor_sync(0xffffffffu, hi ? acc[1] : acc[3], 4);
    double s = (mid ? s1 : s0) + __shfl_xor_sync(0xffffffffu, mid ? s0 : s1, 2);
    s += __shfl_xor_sync(0xffffffffu, s, 1);
    const int64_t row = row0 + (sub >> 1);
    if (!(sub & 1) && row < end) y[row] = s;
}

}  // namespace rsai
