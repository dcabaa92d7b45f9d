// spmv.cuh -- rows of a CSR product, shared by rsai_spmv / rsai_apply and the solver
#pragma once

#include <stdint.h>

namespace rsai {

struct CsrView {
    const int64_t *row_ptr;
    const int32_t *col_idx;
    const double *val;
};

// Entries up to which a row is one of several on its 8 lanes (three rounds of 8 lanes: the
// longest row of M on a stencil has 19, and of A 7)
constexpr int kShortRow = 24;

// The entries sub, sub + 8, .. of a row of `len` at `at`, in order; U of them in flight, and
// the next U read while the products of these wait for x
template <int U>
__device__ __forceinline__ double lane_chain(const CsrView &A, const double *x, int64_t at, int len, int sub) {
    const int32_t *ci = A.col_idx + at;
    const double *va = A.val + at;
    int32_t c[U];
    double v[U], acc = 0.0;
    int e = sub;
    auto load = [&](int32_t (&cn)[U], double (&vn)[U]) {
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const bool in = e + 8 * u < len;
            cn[u] = in ? ci[e + 8 * u] : -1;
            vn[u] = in ? va[e + 8 * u] : 0.0;
        }
    };
    load(c, v);
    while (e < len) {
        double xv[U], vn[U];
        int32_t cn[U];
#pragma unroll
        for (int u = 0; u < U; ++u) xv[u] = c[u] >= 0 ? x[c[u]] : 0.0;
        e += 8 * U;
        load(cn, vn);
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (c[u] >= 0) acc = fma(v[u], xv[u], acc);
#pragma unroll
        for (int u = 0; u < U; ++u) {
            c[u] = cn[u];
            v[u] = vn[u];
        }
    }
    return acc;
}

// y[row] = (A x)[row] on the 8 lanes of a group (`have`: the group has a row); every lane of the warp calls
template <int U>
__device__ __forceinline__ void spmv_row(const CsrView &A, const double *x, double *y, int64_t row, bool have, int sub) {
    double s = 0.0;
    if (have) {
        const int64_t a = A.row_ptr[row];
        s = lane_chain<U>(A, x, a, (int)(A.row_ptr[row + 1] - a), sub);
    }
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (have && sub == 0) y[row] = s;
}

// y[row0 .. row0 + R) = (A x) of these rows (rows >= end: nothing), R = 1, 2 or 4, on the 8
// lanes sub = 0..7 of a group; the four groups of a warp take consecutive rows and every lane
// of the warp calls.  For every R: lane sub of a row adds entries sub, sub + 8, ... in
// order and a butterfly over 4, 2, 1 joins the lanes, so all of them give the same bits.
//
// R > 1 rows of at most kShortRow entries go side by side: their loads (AHEAD: and those of
// the next round of 8 entries) are in flight together, and the butterflies are one
// reduce-scatter (4 additions per lane for four rows instead of 12, the same sums): on
// this GPU's FP64 unit (2 lanes per cycle and SM) the additions of one butterfly per
// row took longer than the products of a row of 16 entries.
// A longer row would hold the others' lanes up; spmv_short_rows leaves it and sets its bit in
// the mask that it returns, and spmv_long_rows takes the warp's long rows one per group (with all
// rows side by side M of a power law, 60000 rows of 69 entries, took 39 us instead of the 28
// of a row per group, and 100000 rows of 9 entries, a few of 200, 26 instead of 16).
template <int R, bool AHEAD = true>
__device__ __forceinline__ unsigned spmv_short_rows(const CsrView &A, const double *x, double *y, int64_t row0,
                                                    int64_t end, int sub) {
    static_assert(R == 2 || R == 4, "the exchanges below");
    int64_t at[R];
    int len[R];
    int most = 0;
    unsigned is_long = 0;
    int64_t a = row0 < end ? A.row_ptr[row0] : 0;
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int64_t b = row0 + r < end ? A.row_ptr[row0 + r + 1] : a;
        at[r] = a;
        len[r] = (int)(b - a);
        if (len[r] > kShortRow) {
            is_long |= 1u << r;
            len[r] = 0;
        }
        most = max(most, len[r]);
        a = b;
    }
    double acc[R];
#pragma unroll
    for (int r = 0; r < R; ++r) acc[r] = 0.0;
    auto load = [&](int e, int32_t (&c)[R], double (&v)[R]) {
#pragma unroll
        for (int r = 0; r < R; ++r) {
            c[r] = e < len[r] ? A.col_idx[at[r] + e] : -1;
            v[r] = e < len[r] ? A.val[at[r] + e] : 0.0;
        }
    };
    auto add = [&](const int32_t (&c)[R], const double (&v)[R]) {
#pragma unroll
        for (int r = 0; r < R; ++r)
            if (c[r] >= 0) acc[r] = fma(v[r], x[c[r]], acc[r]);
    };
    if constexpr (AHEAD) {
        int32_t c[R];
        double v[R];
        load(sub, c, v);
        for (int e = sub; e < most;) {
            e += 8;
            int32_t cn[R];
            double vn[R];
            load(e, cn, vn);
            add(c, v);
#pragma unroll
            for (int r = 0; r < R; ++r) {
                c[r] = cn[r];
                v[r] = vn[r];
            }
        }
    } else {
        for (int e = sub; e < most; e += 8) {
            int32_t c[R];
            double v[R];
            load(e, c, v);
            add(c, v);
        }
    }
    const bool hi = sub & 4, mid = sub & 2;
    double s;
    if constexpr (R == 4) {
        const double s0 = (hi ? acc[2] : acc[0]) + __shfl_xor_sync(0xffffffffu, hi ? acc[0] : acc[2], 4);
        const double s1 = (hi ? acc[3] : acc[1]) + __shfl_xor_sync(0xffffffffu, hi ? acc[1] : acc[3], 4);
        s = (mid ? s1 : s0) + __shfl_xor_sync(0xffffffffu, mid ? s0 : s1, 2);
    } else {
        s = (hi ? acc[1] : acc[0]) + __shfl_xor_sync(0xffffffffu, hi ? acc[0] : acc[1], 4);
        s += __shfl_xor_sync(0xffffffffu, s, 2);
    }
    s += __shfl_xor_sync(0xffffffffu, s, 1);
    const int mine = sub * R / 8;
    if (sub % (8 / R) == 0 && row0 + mine < end && !(is_long >> mine & 1u)) y[row0 + mine] = s;
    return is_long;
}

// The long rows of the warp's groups (is_long: of the calling lane's group, from row0 on), one per group at a time
template <int R>
__device__ __forceinline__ void spmv_long_rows(const CsrView &A, const double *x, double *y, int64_t row0,
                                               unsigned is_long, int sub) {
    // lane 8 g + r votes for row r of group g; group g takes the g-th of the rows left
    const int group = (threadIdx.x >> 3) & 3;
    const int64_t first = row0 - R * group;
    for (unsigned left = __ballot_sync(0xffffffffu, sub < R && (is_long >> sub & 1u)); left;) {
        unsigned w = left;
        for (int g = 0; g < group; ++g) w &= w - 1u;
        const int bit = __ffs(w) - 1;
        spmv_row<4>(A, x, y, first + R * (bit >> 3) + (bit & 7), w != 0u, sub);
        for (int g = 0; g < 4; ++g) left &= left - 1u;
    }
}

// Rows per group for n rows with nnz entries: one where rows are long on the average (rows
// side by side would wait for the longest) or where groups of more would leave SMs idle, four where
// there are warps enough for the FP64 unit to be what bounds it.  Times in us with 1, 2 and 4 (128
// threads per CTA, launches back to back with gaps of about 1 us): 5 entries per row, n = 20000 7.3, 5.3, 5.3, n = 262144 25.8, 15.5, 13.5; 17
// per row, 2000 5.3, 5.3, 7.3, 60000 11.4, 9.4, 9.4, 262144 31.9, 22.2, 21.7; power-law
// rows of 9 on the average, 5000 9.4, 9.4, 9.4, 20000 9.4, 9.4, 11.4, 262144 32.0, 29.8, 30.2;
// rows of 79, 2000 11.4, 13.5, 17.6, 20000 15.5, 17.6, 22.8, 262144 109, 107, 111.
constexpr int64_t kLongAverage = 32;
inline int spmv_rows_per_group(int64_t n, int64_t nnz) {
    if (nnz / (n > 0 ? n : 1) >= kLongAverage || n <= 12288) return 1;
    return n <= 65536 ? 2 : 4;
}

}  // namespace rsai
