// team_qr.cuh -- unblocked Householder QR on one team: the whole solve of the
// warp bins, the factor of the shared-memory CTA bins, and the pieces that the
// blocked version (panel.cuh) falls back to.
#pragma once

#include "common.cuh"

namespace rsai {

// rhs[0..p) <- R^{-1} rhs[0..p) (column-oriented, in place)
template <class Team, typename T>
__device__ void back_substitute_team(const Team &team, const T *B, int q, int p, T *rhs, T small) {
    const int me = team.rank();
    for (int i = p - 1; i >= 0; --i) {
        T d = B[(int64_t)i * q + i];
        T xi = (fabs(d) <= small) ? T(0) : rhs[i] / d;
        team.sync();
        for (int c = me; c < i; c += Team::SIZE) rhs[c] -= B[(int64_t)i * q + c] * xi;
        if (me == 0) rhs[i] = xi;
        team.sync();
    }
}

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
    T part = 0;
    for (int i = j + me; i < q; i += Team::SIZE) part += col[i] * col[i];
    const T sigma = team.sum(part);
    const T x0 = col[j];
    const T nrm = sqrt(sigma);
    const T alpha = (x0 >= T(0)) ? -nrm : nrm;
    const T v0 = x0 - alpha;
    const T vtv = sigma - x0 * x0 + v0 * v0;
    const T two_over = (vtv > T(0)) ? T(2) / vtv : T(0);
    if (two_over > T(0)) {
        for (int c = c_begin + wid; c <= p; c += NW) {
            T *t = (c < p) ? B + (int64_t)c * q : rhs;
            T d = 0;
            for (int i = j + lane; i < q; i += LN) d += ((i == j) ? v0 : col[i]) * t[i];
            d = team.lanes_sum(d);
            const T f = d * two_over;
            for (int i = j + lane; i < q; i += LN) t[i] -= f * ((i == j) ? v0 : col[i]);
        }
    }
    team.sync();
    if (me == 0) {
        col[j] = alpha;
        vhead[j] = v0;
        taus[j] = two_over;
    }
    rank_flag |= (fabs(alpha) <= small) ? 1 : 0;
    team.sync();
}

// Householder QR of B (q x p, column-major, ld q) applied to rhs, then back
// substitution into rhs[0..p).  Keeps the reflectors (v_j below the diagonal
// of B, heads in vhead, tau = 2 / v^T v in tau) for the refinement solve.  Returns the
// rank flag.  Team-generic, one team synchronisation per step; not inlined.
template <class Team, typename T>
__device__ __noinline__ int qr_solve_team(Team team, T *B, int q, int p, T *rhs, T *vhead, T *taus, T small) {
    int rank_flag = 0;
    for (int j = 0; j < p; ++j) householder_step(team, B, q, p, rhs, vhead, taus, j, j + 1, small, rank_flag);
    back_substitute_team(team, B, q, p, rhs, small);
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

// rhs <- Q^T rhs with the stored reflectors, then R^{-1}; not inlined
template <class Team, typename T>
__device__ __noinline__ void apply_qt_team(Team team, const T *B, int q, int p, T *rhs, const T *vhead,
                                           const T *taus, T small) {
    const int me = team.rank();
    for (int j = 0; j < p; ++j) {
        const T *col = B + (int64_t)j * q;
        const T v0 = vhead[j], tau = taus[j];
        if (tau > T(0)) {
            T d = 0;
            for (int i = me; i < q; i += Team::SIZE)
                if (i >= j) d += ((i == j) ? v0 : col[i]) * rhs[i];
            T sdot = team.sum(d);
            T f = sdot * tau;
            for (int i = me; i < q; i += Team::SIZE)
                if (i >= j) rhs[i] -= f * ((i == j) ? v0 : col[i]);
        }
        team.sync();
    }
    if constexpr (is_lane_team<Team>::value) back_substitute_team(team, B, q, p, rhs, small);
    else back_substitute_blocked(team, B, q, p, rhs, small);
}

// Reflector j (built on q0 rows) applied to the columns p0..p-1 of B (ld q),
// one warp per column; ends with a team synchronisation.
template <class Team, typename T>
__device__ __forceinline__ void update_one_reflector(const Team &team, T *B, int q, int p, int q0, int p0,
                                                     const T *vhead, const T *taus, int j) {
    const int me = team.rank();
    const int lane = me & 31, wid = me >> 5;
    constexpr int NW = (Team::SIZE + 31) / 32;
    const T *col = B + (int64_t)j * q;
    const T v0 = vhead[j], two_over = taus[j];
    if (two_over > T(0)) {
        for (int c = p0 + wid; c < p; c += NW) {
            T *t = B + (int64_t)c * q;
            T d = 0;
            for (int i = j + lane; i < q0; i += 32) d += ((i == j) ? v0 : col[i]) * t[i];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) d += __shfl_xor_sync(0xffffffffu, d, o);
            const T f = d * two_over;
            for (int i = j + lane; i < q0; i += 32) t[i] -= f * ((i == j) ? v0 : col[i]);
        }
    }
    team.sync();
}

}  // namespace rsai
