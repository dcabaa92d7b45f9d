// team_qr.cuh -- unblocked Householder QR on one team: the whole solve of the
// warp bins, the factor of the shared-memory CTA bins, and the pieces that the
// blocked version (panel.cuh) falls back to.
#pragma once

#include "common.cuh"

namespace rsai {

// x >= 0, x > 0 and |x| <= y (y >= 0) as the comparisons give them (NaN: false);
// of doubles on their bit patterns, which keeps the FP64 unit free
__device__ __forceinline__ bool not_negative(float x) { return x >= 0.0f; }
__device__ __forceinline__ bool not_negative(double x) {
    const long long b = __double_as_longlong(x);
    return (b >= 0 && b <= 0x7ff0000000000000LL) || b == LLONG_MIN;  // LLONG_MIN: -0.0
}
__device__ __forceinline__ bool positive(float x) { return x > 0.0f; }
__device__ __forceinline__ bool positive(double x) {
    const long long b = __double_as_longlong(x);
    return b > 0 && b <= 0x7ff0000000000000LL;
}
__device__ __forceinline__ bool abs_at_most(float x, float y) { return fabs(x) <= y; }
__device__ __forceinline__ bool abs_at_most(double x, double y) {
    return abskey(x) <= __double_as_longlong(y) && __double_as_longlong(y) <= 0x7ff0000000000000LL;
}

// 2 / x, x > 0.  In FP64 twice the rounded reciprocal, which is the rounded quotient (a
// power of two scales exactly) for three FP64 instructions less; from 2^1021 on, where
// the reciprocal comes near the subnormals and is rounded to fewer bits, the division.
__device__ __forceinline__ float two_over_of(float x) { return 2.0f / x; }
__device__ __forceinline__ double two_over_of(double x) {
    return __double2hiint(x) < 0x7fc00000 ? 2.0 * (1.0 / x) : 2.0 / x;
}

// a / d for several a with one d.  FP64: Markstein's quotient (IBM J. Res. Dev. 34,
// 1990) from the rounded reciprocal r of d, an estimate and one correction by its
// remainder, three FP64 instructions; the plain division where an operand is so
// small or large that one of them could leave the range.  The bits of the division
// in every case: of a zero the estimate, which has the quotient's sign (the
// correction would add +0 to it).
template <typename T> struct Divisor;
template <> struct Divisor<float> {
    float d;
    __device__ __forceinline__ explicit Divisor(float x) : d(x) {}
    __device__ __forceinline__ float into(float a) const { return a / d; }
};
__device__ __forceinline__ bool mid_range(double x) {  // 2^-500 <= |x| < 2^500
    const unsigned e = ((unsigned)__double2hiint(x) >> 20) & 0x7ffu;
    return e - 523u < 1000u;
}
__device__ __forceinline__ bool is_zero(double x) {  // on the bits: the FP64 unit stays free
    return ((unsigned)__double2hiint(x) << 1 | (unsigned)__double2loint(x)) == 0u;
}
template <> struct Divisor<double> {
    double d, r;
    bool mid;
    __device__ __forceinline__ explicit Divisor(double x) : d(x), r(1.0 / x), mid(mid_range(x)) {}
    __device__ __forceinline__ double into(double a) const {
        if (mid && (mid_range(a) || is_zero(a))) {
            const double e = a * r, x = fma(fma(-e, d, a), r, e);
            return is_zero(a) ? e : x;
        }
        return a / d;
    }
};

// Triangular solves on a team within a warp, p <= its lanes: lane c keeps rhs[c], and
// its quotient is formed by every lane beforehand, so that a step is a quotient,
// a shuffle and one fused multiply-add instead of a trip through shared memory with
// two synchronisations.  Bound by that chain, in FP64 also by the quotients (the FP64 unit
// takes 2 lanes per cycle and SM): with Divisor and two_over_of, 64^3 in FP64 15.1 -> 14.2 ms
// and the 40^3 FP64 refit and adjoint 7.9 -> 7.1 ms.
// UP: R x = rhs, from the last row; else R^T y = rhs.
template <bool UP, class Team, typename T>
__device__ __forceinline__ void triangular_lanes(const Team &team, const T *B, int q, int p, T *rhs, T small) {
    const int me = team.rank();
    const bool mine = me < p;
    const T dd = mine ? B[me * q + me] : T(1);
    const bool zero = abs_at_most(dd, small);
    const Divisor<T> div(dd);
    T x = mine ? rhs[me] : T(0);
    const T *row = UP ? B + me : B + (mine ? me : 0) * q;
    const int step = UP ? q : 1;
    for (int t = 0; t < p; ++t) {
        const int i = UP ? p - 1 - t : t;
        const bool below = mine && (UP ? me < i : me > i);
        const T b = below ? row[i * step] : T(0);
        const T xi = team.bcast(zero ? T(0) : div.into(x), i);
        if (below) x -= b * xi;
        else if (me == i) x = xi;
    }
    if (mine) rhs[me] = x;
    team.sync();
}

// rhs <- Q^T rhs with the stored reflectors, then R^{-1}, on a team within a warp:
// rows me, me + W, .. of rhs stay in registers (q <= 4 W in every such bin), and the
// next reflector is read while the dot product of one is reduced (33^3 at eps = 0.15,
// where it is an eighth of the warp bins' time: 29.5 -> 29.0 ms).
template <class Team, typename T>
__device__ __noinline__ void apply_qt_lanes(Team team, const T *B, int q, int p, T *rhs, const T *vhead, const T *taus,
                                            T small) {
    constexpr int W = Team::SIZE, R = 4;
    const int me = team.rank();
    T x[R], vn[R], v0n = vhead[0], taun = taus[0];
#pragma unroll
    for (int u = 0; u < R; ++u) {
        const int i = me + W * u;
        x[u] = i < q ? rhs[i] : T(0);
        vn[u] = i < q ? B[i] : T(0);
    }
    for (int j = 0; j < p; ++j) {
        T v[R];
        const T tau = taun;
#pragma unroll
        for (int u = 0; u < R; ++u) v[u] = me + W * u == j ? v0n : vn[u];
        if (j + 1 < p) {
            v0n = vhead[j + 1];
            taun = taus[j + 1];
#pragma unroll
            for (int u = 0; u < R; ++u) {
                const int i = me + W * u;
                vn[u] = i < q ? B[(j + 1) * q + i] : T(0);
            }
        }
        if (tau > T(0)) {
            T d = T(0);
#pragma unroll
            for (int u = 0; u < R; ++u)
                if (me + W * u >= j && me + W * u < q) d += v[u] * x[u];
            const T f = team.sum(d) * tau;
#pragma unroll
            for (int u = 0; u < R; ++u)
                if (me + W * u >= j) x[u] -= f * v[u];
        }
    }
#pragma unroll
    for (int u = 0; u < R; ++u)
        if (me + W * u < q) rhs[me + W * u] = x[u];
    team.sync();
    triangular_lanes<true>(team, B, q, p, rhs, small);
}

// A Householder update of the M columns c0..c0+M-1 of B (c == p: rhs; past p:
// nothing), rows j..q-1, on W lanes of one warp: t <- t - f v, f = two_over (v . t).
// The dot products are summed over the lanes together: a reduce-scatter leaves
// column u's sum on the lanes u * W / M.., by the additions of M separate
// butterflies but M - 1 + log2(W / M) of them per lane instead of M log2 W, and
// with M chains in flight instead of one.  In FP64 (2 lanes per cycle and SM) the
// additions were as much work as the products: 64^3 in FP64, three rows per lane,
// 11 FP64 instructions per column and step against 7 to 8.
template <int M, int W, typename T>
__device__ __forceinline__ void update_columns(unsigned mask, int lane, T *B, int ld, int q, int p, T *rhs,
                                               const T *col, T v0, T two_over, int j, int c0) {
    T x[M];
    T *t[M];
#pragma unroll
    for (int u = 0; u < M; ++u) {
        x[u] = T(0);
        t[u] = c0 + u < p ? B + (int64_t)(c0 + u) * ld : rhs;
    }
    for (int i = j + lane; i < q; i += W) {
        const T v = (i == j) ? v0 : col[i];
#pragma unroll
        for (int u = 0; u < M; ++u)
            if (c0 + u <= p) x[u] += v * t[u][i];
    }
#pragma unroll
    for (int h = M / 2, o = W / 2; h >= 1; h >>= 1, o >>= 1) {
        const bool up = (lane & o) != 0;
#pragma unroll
        for (int u = 0; u < h; ++u) {
            const T send = up ? x[u] : x[u + h];
            const T keep = up ? x[u + h] : x[u];
            x[u] = keep + __shfl_xor_sync(mask, send, o);
        }
    }
#pragma unroll
    for (int o = W / 2 / M; o > 0; o >>= 1) x[0] += __shfl_xor_sync(mask, x[0], o);
    const T f = x[0] * two_over;
    T fu[M];
#pragma unroll
    for (int u = 0; u < M; ++u) fu[u] = __shfl_sync(mask, f, u * (W / M), W);
    for (int i = j + lane; i < q; i += W) {
        const T v = (i == j) ? v0 : col[i];
#pragma unroll
        for (int u = 0; u < M; ++u)
            if (c0 + u <= p) t[u][i] -= fu[u] * v;
    }
}

// lanes of the calling thread's group of W lanes
template <int W> __device__ __forceinline__ unsigned group_mask() {
    if constexpr (W == 32) return 0xffffffffu;
    else return 0xffffu << (threadIdx.x & 16);
}

// The reflector of a column from its norm^2 and head x0: R_jj, v(j), 2 / v^T v
template <typename T> __device__ __forceinline__ void reflector(T sigma, T x0, T &alpha, T &v0, T &two_over) {
    const T nrm = sqrt(sigma);
    alpha = not_negative(x0) ? -nrm : nrm;
    v0 = x0 - alpha;
    const T vtv = sigma - x0 * x0 + v0 * v0;
    two_over = positive(vtv) ? two_over_of(vtv) : T(0);
}

// This thread's terms of the sum of squares of col[j..q) (BlockTeam::sum_rows)
template <class Team, typename T>
__device__ __forceinline__ void squares_of_rows(const T *col, int j, int q, int me, T (&part)[Team::VK]) {
    if constexpr (Team::VK == 1) {
        part[0] = T(0);
        for (int i = j + me; i < q; i += Team::SIZE) part[0] += col[i] * col[i];
    } else {
#pragma unroll
        for (int v = 0; v < Team::VK; ++v) {
            const int i = j + me + v * Team::SIZE;
            part[v] = i < q ? col[i] * col[i] : T(0);
        }
    }
}

// Columns that a warp's FP32 update takes at a time (33^3 at eps = 0.15: bins W and
// W2 11.5 ms with one, 9.0 with four)
constexpr int kLaneBatch32 = 4;

// One Householder step j on B (q x p, ld q) and rhs: the reflector of column j
// over rows >= j, applied to the columns c in [c_begin, p) and to rhs.  The
// norm is one team reduction; the columns are dealt out to the team's warps,
// each warp forming its column's dot product (lanes over rows, one warp
// reduction) and applying the update itself.  Stores R_jj, v_j(j), v_j^T v_j.
template <class Team, typename T>
__device__ __forceinline__ void householder_step(const Team &team, T *B, int q, int p, T *rhs, T *vhead, T *taus,
                                                 int j, int c_begin, T small, int &rank_flag) {
    const int me = team.rank();
    constexpr int LN = Team::LANES;  // lanes of one group: the team itself, or one warp of a CTA
    constexpr int NW = Team::SIZE / LN;
    const int lane = me % LN, wid = me / LN;
    T *col = B + (int64_t)j * q;
    T alpha, v0, two_over;
    if constexpr (!is_lane_team<Team>::value && sizeof(T) == 8) {
        // the warps' sums, the square root and the division on one warp: as
        // much FP64 work per warp as the update of several columns
        constexpr int VK = Team::VK;
        T part[VK];
        squares_of_rows<Team>(col, j, q, me, part);
#pragma unroll
        for (int v = 0; v < VK; ++v) part[v] = team.lanes_sum(part[v]);
        team.sync();
        if (lane == 0) {
#pragma unroll
            for (int v = 0; v < VK; ++v) team.template slot<T>(wid + NW * v) = part[v];
        }
        team.sync();
        if (wid == 0) {
            T sigma = team.template slot<T>(0);
#pragma unroll
            for (int w = 1; w < NW * VK; ++w) sigma += team.template slot<T>(w);
            reflector(sigma, col[j], alpha, v0, two_over);
            __syncwarp();
            if (lane == 0) {
                team.template slot<T>(0) = alpha;
                team.template slot<T>(1) = v0;
                team.template slot<T>(2) = two_over;
            }
        }
        team.sync();
        alpha = team.template slot<T>(0);
        v0 = team.template slot<T>(1);
        two_over = team.template slot<T>(2);
    } else if constexpr (!is_lane_team<Team>::value) {
        T part[Team::VK];
        squares_of_rows<Team>(col, j, q, me, part);
        reflector(team.sum_rows(part), col[j], alpha, v0, two_over);
    } else {
        T part = 0;
        for (int i = j + me; i < q; i += Team::SIZE) part += col[i] * col[i];
        reflector(team.sum(part), col[j], alpha, v0, two_over);
    }
    if (positive(two_over)) {
        const unsigned mask = group_mask<LN>();
        if constexpr (is_lane_team<Team>::value && sizeof(T) == 4) {
            for (int c = c_begin; c <= p; c += kLaneBatch32)
                update_columns<kLaneBatch32, LN>(mask, lane, B, q, q, p, rhs, col, v0, two_over, j, c);
        } else if constexpr (is_lane_team<Team>::value) {
            int c = c_begin;
            for (; c + 4 <= p; c += 8) update_columns<8, LN>(mask, lane, B, q, q, p, rhs, col, v0, two_over, j, c);
            if (c + 1 < p) {
                update_columns<4, LN>(mask, lane, B, q, q, p, rhs, col, v0, two_over, j, c);
                c += 4;
            }
            for (; c <= p; c += 2) update_columns<2, LN>(mask, lane, B, q, q, p, rhs, col, v0, two_over, j, c);
        } else {
            // an even share per warp, four or two or one at a time
            const int left = p - c_begin + 1;
            if (left > 2 * NW) {
                for (int c = c_begin + 4 * wid; c <= p; c += 4 * NW)
                    update_columns<4, LN>(mask, lane, B, q, q, p, rhs, col, v0, two_over, j, c);
            } else if (left > NW) {
                for (int c = c_begin + 2 * wid; c <= p; c += 2 * NW)
                    update_columns<2, LN>(mask, lane, B, q, q, p, rhs, col, v0, two_over, j, c);
            } else if (c_begin + wid <= p) {
                update_columns<1, LN>(mask, lane, B, q, q, p, rhs, col, v0, two_over, j, c_begin + wid);
            }
        }
    }
    team.sync();
    if (me == 0) {
        col[j] = alpha;
        vhead[j] = v0;
        taus[j] = two_over;
    }
    rank_flag |= abs_at_most(alpha, small) ? 1 : 0;
    team.sync();
}

// Householder QR of B (q x p, column-major, ld q) applied to rhs, then back
// substitution into rhs[0..p), on a team within a warp.  Keeps the reflectors (v_j below
// the diagonal of B, heads in vhead, tau = 2 / v^T v in tau) for the refinement solve.
// Returns the rank flag.  Not inlined.
template <class Team, typename T>
__device__ __noinline__ int qr_solve_team(Team team, T *B, int q, int p, T *rhs, T *vhead, T *taus, T small) {
    int rank_flag = 0;
    for (int j = 0; j < p; ++j) householder_step(team, B, q, p, rhs, vhead, taus, j, j + 1, small, rank_flag);
    triangular_lanes<true>(team, B, q, p, rhs, small);
    return rank_flag;
}

// Householder steps j_start..p-1 on B and rhs, no back substitution (rhs is
// left holding Q^T rhs): a factor from scratch (j_start = 0) that is kept for
// later updates, or the appended block of the QR update.  Not inlined.
template <class Team, typename T>
__device__ __noinline__ int qr_factor_team(Team team, T *B, int q, int p, T *rhs, T *vhead, T *taus, T small,
                                           int j_start) {
    int rank_flag = 0;
    for (int j = j_start; j < p; ++j) householder_step(team, B, q, p, rhs, vhead, taus, j, j + 1, small, rank_flag);
    return rank_flag;
}

// rhs[0..p) <- R^{-1} rhs[0..p) for a CTA team, in blocks of kBS rows from
// the bottom: one warp solves the block's triangle (lane l holds row b0 + l
// and loads its row of the block into registers first), then every thread
// subtracts the block's part from the rows above.  Each row receives its
// terms in the same order (descending column) as the one-row-at-a-time
// version, so the results are identical.
template <class Team, typename T>
__device__ void back_substitute_blocked(const Team &team, const T *B, int q, int p, T *rhs, T small) {
    constexpr int kBS = sizeof(T) == 8 ? 16 : 32;
    const int me = team.rank();
    for (int b1 = p; b1 > 0;) {
        const int b0 = max(0, b1 - kBS);
        const int nbk = b1 - b0;
        if (me < 32) {
            const int i = b0 + me;
            const bool row = me < nbk;
            T rv[kBS];
#pragma unroll
            for (int u = 0; u < kBS; ++u) rv[u] = (row && u < nbk) ? B[(int64_t)(b0 + u) * q + i] : T(0);
            const T dd = row ? B[(int64_t)i * q + i] : T(1);
            T xi = row ? rhs[i] : T(0);
#pragma unroll
            for (int u = kBS - 1; u >= 0; --u) {
                if (u < nbk) {
                    const T rr = __shfl_sync(0xffffffffu, xi, u);
                    const T d = __shfl_sync(0xffffffffu, dd, u);
                    const T xr = (fabs(d) <= small) ? T(0) : rr / d;
                    if (me == u) xi = xr;
                    else if (me < u) xi -= rv[u] * xr;
                }
            }
            if (row) rhs[i] = xi;
        }
        team.sync();
        for (int c = me; c < b0; c += Team::SIZE) {
            T bv[kBS];
#pragma unroll
            for (int u = 0; u < kBS; ++u) bv[u] = (u < nbk) ? B[(int64_t)(b0 + u) * q + c] : T(0);
            T a = rhs[c];
#pragma unroll
            for (int u = kBS - 1; u >= 0; --u)
                if (u < nbk) a -= bv[u] * rhs[b0 + u];
            rhs[c] = a;
        }
        team.sync();
        b1 = b0;
    }
}

// rhs[0..p) <- R^{-T} rhs[0..p) for a CTA team, in blocks of kBS rows from the top:
// one warp solves the block's triangle (lane l holds row b0 + l), then every
// thread subtracts the block's part from a row below, in the order of one row
// at a time (the same bits).  Row c of R^T is column c of B: with B in global memory
// (stage != NULL) the block's kBS entries of each column are copied to
// the staging area first, a warp per column, as many columns at a time as fit.
// One row at a time it took two synchronisations and a strided load per row.
template <class Team, typename T>
__device__ __noinline__ void forward_substitute_blocked(Team team, const T *B, int q, int p, T *rhs, T small, T *stage,
                                                        int stage_bytes) {
    constexpr int kBS = sizeof(T) == 8 ? 16 : 32, LD = kBS + 1;
    const int me = team.rank();
    const int chunk = Team::STAGED ? stage_bytes / (int)(LD * sizeof(T)) : p;
    for (int b0 = 0; b0 < p; b0 += kBS) {
        const int nbk = min(kBS, p - b0);
        for (int c0 = b0; c0 < p; c0 += chunk) {
            const int c1 = min(p, c0 + chunk);
            if constexpr (Team::STAGED) {
                for (int e = me; e < (c1 - c0) * kBS; e += Team::SIZE) {
                    const int c = e / kBS, u = e % kBS;
                    if (u < nbk) stage[c * LD + u] = B[(int64_t)(c0 + c) * q + b0 + u];
                }
                team.sync();
            }
            auto entry = [&](int c, int u) {  // R(b0 + u, c)
                if constexpr (Team::STAGED) return stage[(c - c0) * LD + u];
                else return B[(int64_t)c * q + b0 + u];
            };
            if (c0 == b0 && me < 32) {
                const bool row = me < nbk;
                T rv[kBS];
#pragma unroll
                for (int u = 0; u < kBS; ++u) rv[u] = (row && u < me) ? entry(b0 + me, u) : T(0);
                const T dd = row ? entry(b0 + me, me) : T(1);
                T yi = row ? rhs[b0 + me] : T(0);
#pragma unroll
                for (int u = 0; u < kBS; ++u) {
                    if (u < nbk) {
                        const T a = __shfl_sync(0xffffffffu, yi, u);
                        const T d = __shfl_sync(0xffffffffu, dd, u);
                        const T y = (fabs(d) <= small) ? T(0) : a / d;
                        if (me == u) yi = y;
                        else if (me > u) yi -= rv[u] * y;
                    }
                }
                if (row) rhs[b0 + me] = yi;
            }
            team.sync();
            for (int c = max(c0, b0 + nbk) + me; c < c1; c += Team::SIZE) {
                T a = rhs[c];
                for (int u = 0; u < nbk; ++u) a -= entry(c, u) * rhs[b0 + u];
                rhs[c] = a;
            }
            team.sync();
        }
    }
}

// rhs <- Q^T rhs with the stored reflectors, then R^{-1}, on a CTA; not inlined
template <class Team, typename T>
__device__ __noinline__ void apply_qt_team(Team team, const T *B, int q, int p, T *rhs, const T *vhead,
                                           const T *taus, T small) {
    const int me = team.rank();
    for (int j = 0; j < p; ++j) {
        const T *col = B + (int64_t)j * q;
        const T v0 = vhead[j], tau = taus[j];
        if (tau > T(0)) {
            T d[Team::VK];
#pragma unroll
            for (int v = 0; v < Team::VK; ++v) {
                d[v] = T(0);
                for (int i = me + v * Team::SIZE; i < q; i += Team::VK == 1 ? Team::SIZE : q)
                    if (i >= j) d[v] += ((i == j) ? v0 : col[i]) * rhs[i];
            }
            const T f = team.sum_rows(d) * tau;
            for (int i = me; i < q; i += Team::SIZE)
                if (i >= j) rhs[i] -= f * ((i == j) ? v0 : col[i]);
        }
        team.sync();
    }
    back_substitute_blocked(team, B, q, p, rhs, small);
}

// The reflectors j0..j1-1 (built on q0 rows) applied in order to the columns
// p0..p-1 of B (ld q).  A warp takes its columns through all of them, so nothing
// is synchronised until the end.
// M columns per warp at a time.
template <int M, class Team, typename T>
__device__ __forceinline__ void update_reflectors_m(const Team &team, T *B, int q, int p, int q0, int p0,
                                                    const T *vhead, const T *taus, int j0, int j1) {
    const int lane = team.rank() & 31, wid = team.rank() >> 5;
    constexpr int NW = Team::SIZE / 32;
    for (int c = p0 + M * wid; c < p; c += M * NW) {
        for (int j = j0; j < j1; ++j) {
            const T two_over = taus[j];
            // p - 1: the last column is not a right-hand side here
            if (positive(two_over))
                update_columns<M, 32>(0xffffffffu, lane, B, q, q0, p - 1, B + (int64_t)(p - 1) * q, B + (int64_t)j * q,
                                      vhead[j], two_over, j, c);
            __syncwarp();
        }
    }
    team.sync();
}
// Two columns share the loads of a reflector, but are twice as long a chain: with at most one
// column per warp (SPAI appends c at a time) one each (SPAI on the n = 20000 power law in FP64:
// global bin 136 ms with two, 129 with one).
template <class Team, typename T>
__device__ __forceinline__ void update_reflectors(const Team &team, T *B, int q, int p, int q0, int p0,
                                                  const T *vhead, const T *taus, int j0, int j1) {
    if (p - p0 <= Team::SIZE / 32) update_reflectors_m<1>(team, B, q, p, q0, p0, vhead, taus, j0, j1);
    else update_reflectors_m<2>(team, B, q, p, q0, p0, vhead, taus, j0, j1);
}

}  // namespace rsai
