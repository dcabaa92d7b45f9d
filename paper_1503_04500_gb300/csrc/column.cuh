// column.cuh -- one column of RSAI(tol) on one team (warp or CTA).
//
// Per column k (Section 3 Algorithm 1, Section 4 Eq. 4.3):
//   J = {k}, R = {}, l = 0
//   solve(J); drop(J); r = A m - e_k on S = I u {k}; rho = ||r||
//   while rho > eps and l < l_max:
//     Rhat = top-c of {i in S : |r_i| > band, i not in R} by (|r_i| desc, i asc)
//            with a tie band; R += Rhat                        (Eq. 3.2)
//     Jhat = cols(A(Rhat,:)) \ J
//     l += 1; if Jhat is empty: continue
//     J += Jhat; solve(J); drop(J); residual                   (Eq. 4.3)
//
// solve(J): I = rows of A(:,J) (Section 2), B = A(I,J) gathered into the team's
// workspace (column-major, leading dimension q), e = e_k(I), Householder QR of
// B applied to e, back substitution (Eq. 2.3).  In RSAI_FP32_REFINE the QR runs
// in float; the residual of the float solution is formed in double from the
// sparse columns of A, one correction is solved with the float factors and
// added in double.  The residual r_k, its norm, the dominant-row choice, the
// drop test and the stopping test are double in both precisions.
//
// A column whose problem outgrows the team's workspace returns OVERFLOW; the
// caller hands it to the next (larger) bin, which restarts it from J = {k}.
#pragma once

#include <type_traits>

#include "panel.cuh"
#include "stage_map.cuh"
#include "warp_small.cuh"

namespace rsai {

struct Caps {
    int qcap;      // max |I| (rows of the LS problem); |S| <= qcap + 1
    int pcap;      // max |J|
    int scap;      // sort buffer (power of two)
    int rcap;      // max |R| (dominant rows used so far)
    int64_t bcap;  // max q*p elements of B
    int small_p;   // largest |J| solved by the register-resident warp QR (0: never)
    int stage_bytes;  // shared memory for staging QR panels (global-memory bins), 0 = none
    int append;       // CTA bins: room for the kept factor's positions (Section 3)
    int dcap;         // max number of distinct columns dropped from J (they are not charged again on re-entry)
    int spai;         // SPAI selection: a score per candidate column (scap of them)
};

// Caps of a bin whose sizes are fixed at compile time (no SPAI scores): every address in its workspace is then the warp's base plus a constant, and
// the workspace is known to be shared memory.
template <int Q, int P, int S, int R, int D, int APPEND = 0> struct FixedCaps {
    static constexpr int qcap = Q, pcap = P, scap = S, rcap = R, dcap = D;
    static constexpr int64_t bcap = (int64_t)Q * P;
    static constexpr int stage_bytes = 0, append = APPEND, spai = 0;
    int small_p;
    // a frozen pass uses neither the set R nor SPAI's scores
    static bool fits_frozen(const Caps &c) {
        return c.qcap == Q && c.pcap == P && c.scap == S && c.dcap == D && c.bcap == bcap &&
               c.stage_bytes == 0 && c.append == APPEND;
    }
    static bool fits(const Caps &c) { return fits_frozen(c) && c.rcap == R && c.spai == 0; }
};

template <typename T> struct Work {
    T *B, *vhead, *tau, *rhs;
    double *m, *r, *z, *wv;
    long long *ctr;
    int32_t *I, *S, *J, *Jn, *Rset, *buf, *buf2, *Rhat;
    int32_t *D;        // columns dropped from J so far, ascending
    double *sc;        // SPAI: the score s_j of each candidate (Caps::spai)
    int32_t *Ip, *Jp;  // factor position of each sorted I / J entry (Caps::append)
    T *qte;            // Q^T e_k(I) of the kept factor, factor row order (Caps::append)
    // Warp bins: A(I,J) by rows.  Row i of I holds the columns c of J whose bit is
    // set in rmask[i], ascending; their values in double are the entries
    // rstart[i], .. of row_vals(), which shares its memory with buf and buf2 and
    // is valid from a solve until the next use of these.
    uint32_t *rmask;
    int32_t *rstart;
    __device__ __forceinline__ double *row_vals() const { return reinterpret_cast<double *>(buf); }
    // Global-memory bins (Caps::stage_bytes > 0): the reflectors as factored,
    // in panels: pnb[j0] reflectors start at j0, and column j of the panel's
    // compact-WY T (H_j0 ... H_j0+nb-1 = I - V T V^T) is Tst[j * kPanel + s],
    // s <= j - j0.  A reflector factored on its own is a panel of one, T = tau.
    T *Tst;
    int32_t *pnb;
    // not part of the carved workspace (global-memory bins):
    char *stage = nullptr;    // panel staging area (shared memory)
    HelpOwner *ho = nullptr;  // sharing of the trailing updates

    __host__ __device__ static constexpr size_t align16(size_t x) { return (x + 15) & ~size_t(15); }
    template <class CapT> __host__ __device__ static constexpr size_t bytes(const CapT &c) {
        size_t b = 0;
        b += align16(sizeof(T) * (size_t)c.bcap);
        b += 2 * align16(sizeof(T) * (size_t)c.pcap);
        b += align16(sizeof(T) * (size_t)(c.qcap + 1));
        b += align16(sizeof(double) * (size_t)c.pcap);
        b += align16(sizeof(double) * (size_t)(c.qcap + 1));
        b += align16(sizeof(double) * (size_t)c.pcap);
        b += align16(sizeof(double) * (size_t)(c.qcap + 1));
        b += align16(sizeof(long long) * CTR_COUNT);
        b += align16(sizeof(int32_t) * (size_t)c.qcap);
        b += align16(sizeof(int32_t) * (size_t)(c.qcap + 1));
        b += 2 * align16(sizeof(int32_t) * (size_t)c.pcap);
        b += align16(sizeof(int32_t) * (size_t)c.rcap);
        b += 2 * align16(sizeof(int32_t) * (size_t)c.scap);
        b += align16(sizeof(int32_t) * 32);
        b += align16(sizeof(int32_t) * (size_t)c.dcap);
        if (c.spai) b += align16(sizeof(double) * (size_t)c.scap);
        if (c.append) {
            b += align16(sizeof(int32_t) * (size_t)c.qcap);
            b += align16(sizeof(int32_t) * (size_t)c.pcap);
            b += align16(sizeof(T) * (size_t)(c.qcap + 1));
        } else {
            b += 2 * align16(sizeof(int32_t) * (size_t)c.qcap);
        }
        if (c.stage_bytes > 0) {
            b += align16(sizeof(T) * (size_t)c.pcap * kPanel);
            b += align16(sizeof(int32_t) * (size_t)c.pcap);
        }
        return b;
    }
    template <class CapT> __device__ __forceinline__ void carve(char *base, const CapT &c) {
        size_t o = 0;
        B = (T *)(base + o); o += align16(sizeof(T) * (size_t)c.bcap);
        vhead = (T *)(base + o); o += align16(sizeof(T) * (size_t)c.pcap);
        tau = (T *)(base + o); o += align16(sizeof(T) * (size_t)c.pcap);
        rhs = (T *)(base + o); o += align16(sizeof(T) * (size_t)(c.qcap + 1));
        m = (double *)(base + o); o += align16(sizeof(double) * (size_t)c.pcap);
        r = (double *)(base + o); o += align16(sizeof(double) * (size_t)(c.qcap + 1));
        z = (double *)(base + o); o += align16(sizeof(double) * (size_t)c.pcap);
        wv = (double *)(base + o); o += align16(sizeof(double) * (size_t)(c.qcap + 1));
        ctr = (long long *)(base + o); o += align16(sizeof(long long) * CTR_COUNT);
        I = (int32_t *)(base + o); o += align16(sizeof(int32_t) * (size_t)c.qcap);
        S = (int32_t *)(base + o); o += align16(sizeof(int32_t) * (size_t)(c.qcap + 1));
        J = (int32_t *)(base + o); o += align16(sizeof(int32_t) * (size_t)c.pcap);
        Jn = (int32_t *)(base + o); o += align16(sizeof(int32_t) * (size_t)c.pcap);
        Rset = (int32_t *)(base + o); o += align16(sizeof(int32_t) * (size_t)c.rcap);
        buf = (int32_t *)(base + o); o += align16(sizeof(int32_t) * (size_t)c.scap);
        buf2 = (int32_t *)(base + o); o += align16(sizeof(int32_t) * (size_t)c.scap);
        Rhat = (int32_t *)(base + o); o += align16(sizeof(int32_t) * 32);
        D = (int32_t *)(base + o); o += align16(sizeof(int32_t) * (size_t)c.dcap);
        sc = nullptr;
        if (c.spai) {
            sc = (double *)(base + o); o += align16(sizeof(double) * (size_t)c.scap);
        }
        Ip = Jp = nullptr;
        qte = nullptr;
        if (c.append) {
            Ip = (int32_t *)(base + o); o += align16(sizeof(int32_t) * (size_t)c.qcap);
            Jp = (int32_t *)(base + o); o += align16(sizeof(int32_t) * (size_t)c.pcap);
            qte = (T *)(base + o); o += align16(sizeof(T) * (size_t)(c.qcap + 1));
        }
        rmask = nullptr;
        rstart = nullptr;
        if (!c.append) {
            rmask = (uint32_t *)(base + o); o += align16(sizeof(int32_t) * (size_t)c.qcap);
            rstart = (int32_t *)(base + o); o += align16(sizeof(int32_t) * (size_t)c.qcap);
        }
        Tst = nullptr;
        pnb = nullptr;
        if (c.stage_bytes > 0) {
            Tst = (T *)(base + o); o += align16(sizeof(T) * (size_t)c.pcap * kPanel);
            pnb = (int32_t *)(base + o); o += align16(sizeof(int32_t) * (size_t)c.pcap);
        }
    }
};

// COL_OVERFLOW_J: |J| outgrew the bin (a bin with the same |J| limit cannot take the column either)
enum ColStatus { COL_DONE = 0, COL_OVERFLOW = 1, COL_OVERFLOW_J = 2 };

// Rows per lane of the register QR: q <= 64 on a warp, q <= 48 on half a warp
template <class Team> constexpr int kRegRows = Team::SIZE == 16 ? 3 : 2;

// Sort buf[0..len) ascending: registers and shuffles on a warp or half warp
// (up to 256 elements), bitonic in shared memory otherwise.
template <class Team>
__device__ void team_sort_i32(const Team &team, int32_t *buf, int len) {
    if constexpr (is_lane_team<Team>::value) {
        constexpr int W = Team::SIZE;
        if (len <= W) { lanes_sort_regs<W, 1>(buf, len); return; }
        if (len <= 2 * W) { lanes_sort_regs<W, 2>(buf, len); return; }
        if (len <= 4 * W) { lanes_sort_regs<W, 4>(buf, len); return; }
        if (len <= 8 * W) { lanes_sort_regs<W, 8>(buf, len); return; }
        if constexpr (W == 16) {
            if (len <= 16 * W) { lanes_sort_regs<W, 16>(buf, len); return; }
        }
    }
    team_sort_i32_smem(team, buf, len);
}

__host__ __device__ inline int next_pow2(int x) {
    int n = 1;
    while (n < x) n <<= 1;
    return n;
}

// Algorithmic flops of one solve on (q,p) appended to a factorisation of
// (q0,p0) (p0 = 0: from scratch): the reflectors of the old columns applied to
// the new ones, Householder steps p0..p-1 on the stacked rows (norm, then every
// trailing column and the right-hand side), and the back substitution.
__device__ __forceinline__ long long solve_flops(long long q0, long long p0, long long q, long long p) {
    long long mm = p - p0;
    long long f = 4 * mm * (p0 * q0 - p0 * (p0 - 1) / 2);
    long long s2 = mm * (mm + 1) * (2 * mm + 1) / 6;
    f += (q - p) * (2 * mm + 2 * mm * (mm + 1)) + mm * (mm + 1) + 4 * s2;
    return f + p * p;
}

// J = rows of A(:,k), ascending as the CSC keeps them; returns |J|, or -1 if
// it exceeds pcap, and in *bytes the algorithmic bytes of J's columns (12 per
// nonzero + 16 each).  Kept out of line: only the initial pattern of A uses it.
template <class Team>
__device__ __noinline__ int pattern_of_column(Team team, const int64_t *col_ptr, const int32_t *row_idx, int32_t k,
                                              int pcap, int32_t *J, long long *bytes) {
    const int me = team.rank();
    const int64_t e0 = col_ptr[k];
    const int len = (int)(col_ptr[k + 1] - e0);
    if (len > pcap) return -1;
    long long b = 0;
    for (int c = me; c < len; c += Team::SIZE) {
        const int32_t j = row_idx[e0 + c];
        J[c] = j;
        b += 12 * (col_ptr[j + 1] - col_ptr[j]) + 16;
    }
    *bytes = team.sum(b);
    team.sync();
    return len;
}

// J -> position in J, by a binary search of the sorted J
struct JSet {
    const int32_t *J;
    int p;
    __device__ __forceinline__ int find(int32_t col) const { return find_i32(J, p, col); }
};

struct SpaiPick {
    int na;               // columns chosen (in buf, ascending); 0: no candidate; -1: overflow
    long long bytes, sel; // algorithmic bytes and selection flops
};

// SPAI's most profitable indices (Section 2, Eqs. 2.5-2.7).  L = rows of S
// with |r_i| > band (the same reading of r_i != 0 as the dominant rows);
// the candidates Jhat = cols(A(L,:)) \ J, each scored by one rank walking
// its CSC column: s_j = (r^T A e_j)^2 / ||A e_j||^2 in double (rho_j^2 =
// ||r||^2 - s_j, so the largest s_j are the smallest rho_j); the c best by
// (s_j desc, j asc) with a tie band of tie_band * ||r||^2, the scores
// compared as ordered integer keys (non-negative doubles).  The chosen
// columns go to buf in ascending order.  Returns their number, 0 when no
// candidate is left, -1 on overflow.
template <class Team>
__device__ __noinline__ SpaiPick spai_select(Team team, DevA A, int c, double tie_band, int scap, const int32_t *S,
                                             const double *r, int s, JSet Jset, int32_t *buf, int32_t *buf2,
                                             double *sc, int32_t *Rhat) {
    const int me = team.rank();
    SpaiPick out{0, 0, 0};
    long long rinf = 0;
    double rr = 0.0;
    for (int i = me; i < s; i += Team::SIZE) {
        rinf = max(rinf, abskey(r[i]));
        rr = fma(r[i], r[i], rr);
    }
    rinf = team.maxv(rinf);
    rr = team.sum(rr);
    const long long bk = abskey(tie_band * key_value(rinf));
    // column indices of the rows of L
    int tot = 0;
    long long byt = 0;
    for (int i0 = 0; i0 < s; i0 += Team::SIZE) {
        const int i = i0 + me;
        int len = 0;
        int64_t st = 0;
        if (i < s && abskey(r[i]) > bk) {
            const int32_t row = S[i];
            st = A.row_ptr[row];
            len = counted_entries(A.row_ptr[row + 1] - st, scap);
            byt += 4LL * len + 16;
        }
        int part;
        const int off = tot + team.scan(len, &part);
        if (tot + part > scap) {
            out.na = -1;
            return out;
        }
        for (int e = 0; e < len; ++e) buf[off + e] = A.col_idx[st + e];
        tot += part;
    }
    out.bytes += team.sum(byt);
    team.sync();
    if (tot == 0) return out;
    team_sort_i32(team, buf, tot);
    const int nu = team_unique_i32(team, buf, tot, buf2);
    int nc = 0;
    for (int i0 = 0; i0 < nu; i0 += Team::SIZE) {
        const int i = i0 + me;
        const int f = (i < nu) && (Jset.find(buf2[i]) < 0);
        int part;
        const int pos = team.scan(f, &part);
        if (f) buf[nc + pos] = buf2[i];
        nc += part;
    }
    team.sync();
    if (nc == 0) return out;
    // scores (Eq. 2.7)
    long long sf = 0;
    byt = 0;
    for (int t = me; t < nc; t += Team::SIZE) {
        const int32_t j = buf[t];
        double dot = 0.0, nrm = 0.0;
        const int64_t e0 = A.col_ptr[j], e1 = A.col_ptr[j + 1];
        for (int64_t e = e0; e < e1; ++e) {
            const double a = A.cval[e];
            const int pos = find_i32(S, s, A.row_idx[e]);
            if (pos >= 0) dot = fma(r[pos], a, dot);
            nrm = fma(a, a, nrm);
        }
        sc[t] = (nrm > 0.0) ? dot * dot / nrm : 0.0;
        sf += 4 * (e1 - e0) + 3;
        byt += 12 * (e1 - e0) + 16;
    }
    out.sel += team.sum(sf);
    out.bytes += team.sum(byt);
    team.sync();
    const bool take_all = nc <= c;
    long long hik = 0, lob = 0;
    if (!take_all) {
        // the c-th score of the (s_j desc, j asc) order: c rounds of argmax
        long long pa = LLONG_MAX;
        int pi = -1;
        for (int t = 0; t < c; ++t) {
            long long ba = -1;
            int bi = INT32_MAX;
            for (int u = me; u < nc; u += Team::SIZE) {
                const long long a = abskey(sc[u]);
                const int32_t j = buf[u];
                if (dom_before(pa, pi, a, j) && dom_before(a, j, ba, bi)) {
                    ba = a;
                    bi = j;
                }
            }
            team.argmax(ba, bi);
            pa = ba;
            pi = bi;
        }
        const double v = key_value(pa), sband = tie_band * rr;
        hik = abskey(v + sband);
        lob = __double_as_longlong(v - sband);  // negative bit pattern if v - sband < 0
    }
    int nabove = 0;
    if (!take_all) {
        for (int u = me; u < nc; u += Team::SIZE) nabove += abskey(sc[u]) > hik;
        nabove = team.sum(nabove);
    }
    const int need = c - nabove;
    int na = 0, tb = 0;
    for (int u0 = 0; u0 < nc; u0 += Team::SIZE) {
        const int u = u0 + me;
        int above = 0, tie = 0;
        if (u < nc && !take_all) {
            const long long a = abskey(sc[u]);
            above = a > hik;
            tie = (a >= lob) && (a <= hik);
        }
        int tpart;
        const int trank = team.scan(tie, &tpart);
        const int sel = (u < nc) && (take_all || above || (tie && tb + trank < need));
        int part;
        const int pos = team.scan(sel, &part);
        if (sel) Rhat[na + pos] = buf[u];
        na += part;
        tb += tpart;
    }
    team.sync();
    for (int t = me; t < na; t += Team::SIZE) buf[t] = Rhat[t];
    team.sync();
    out.na = na;
    return out;
}


template <class Team, typename T, class CapT = Caps> struct Column {
    const Team &team;
    const DevA &A;
    const DevParams &P;
    const CapT &cap;
    Work<T> &w;
    int32_t k;
    int p, q, s, nR, l, nD;
    int need;  // |J| that did not fit (COL_OVERFLOW_J)
    int64_t q0, p0;
    int rank_flag;
    double rho;
    T small_last;  // rank threshold of the last solve (reused by the adjoint)
    T fro2_f;      // ||B||_F^2 of the kept factor (Caps::append)
    bool fact_valid;  // B, vhead, tau, qte, Ip, Jp hold the factor of the current J (Caps::append)
    // per-column work counters (integers; committed only when the column finishes)
    long long c_qr, c_res, c_ref, c_ref64, c_bytes, c_sel;
    int c_solves, c_drops, c_pmax, c_qmax;

    __device__ Column(const Team &t, const DevA &a, const DevParams &pp, const CapT &c, Work<T> &ww, int32_t kk)
        : team(t), A(a), P(pp), cap(c), w(ww), k(kk) {}

    __device__ __forceinline__ JSet jset() const { return JSet{w.J, p}; }
    __device__ __forceinline__ int find_J(int32_t col) const { return jset().find(col); }

    // The bitmap over indices 0..n-1 in the staging area (global-memory bins;
    // off elsewhere and for n too large for it)
    __device__ __forceinline__ StageMap stage_map() const { return StageMap(w.stage, cap.stage_bytes, A.n); }

    // I = sorted rows of A(:,J) (Section 2).  Returns false on overflow.  In the
    // global-memory bins the staging area keeps the map of I for the gathers.
    __device__ bool rows_of_J() {
        if constexpr (Team::STAGED) {
            const StageMap map = stage_map();
            if (map.on()) {
                map.clear(team);
                int entries = 0;
                for (int c = team.rank(); c < p; c += Team::SIZE) {
                    const int64_t st = A.col_ptr[w.J[c]];
                    const int len = counted_entries(A.col_ptr[w.J[c] + 1] - st, cap.scap);
                    entries += len;
                    for (int e = 0; e < len; e += 4) {
                        int32_t v[4];
#pragma unroll
                        for (int u = 0; u < 4; ++u) v[u] = (e + u < len) ? A.row_idx[st + e + u] : 0;
#pragma unroll
                        for (int u = 0; u < 4; ++u)
                            if (e + u < len) map.mark(v[u]);
                    }
                }
                entries = team.sum(entries);
                const int nq = map.finish(team, w.I, cap.qcap);
                if (entries > cap.scap || nq > cap.qcap) return false;
                q = nq;
                return true;
            }
        }
        int base = 0;
        for (int c0 = 0; c0 < p; c0 += Team::SIZE) {
            int c = c0 + team.rank();
            int len = 0;
            int64_t st = 0;
            if (c < p) {
                st = A.col_ptr[w.J[c]];
                len = counted_entries(A.col_ptr[w.J[c] + 1] - st, cap.scap);
            }
            int tot;
            int off = team.scan(len, &tot);
            if (base + tot > cap.scap) return false;
            for (int e = 0; e < len; e += 4) {
                int32_t v[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) v[u] = (e + u < len) ? A.row_idx[st + e + u] : 0;
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    if (e + u < len) w.buf[base + off + e + u] = v[u];
            }
            base += tot;
        }
        team.sync();
        team_sort_i32(team, w.buf, base);
        int nq = team_unique_i32(team, w.buf, base, w.buf2);
        if (nq > cap.qcap) return false;
        for (int i = team.rank(); i < nq; i += Team::SIZE) w.I[i] = w.buf2[i];
        q = nq;
        team.sync();
        return true;
    }

    // Householder QR of B (q x p, ld q) applied to rhs, then back substitution
    // into rhs[0..p); the reflectors stay in B (tails), vhead and tau.
    __device__ void qr_solve(T small) {
        if constexpr (is_lane_team<Team>::value) {
            if (p > 2 && p <= cap.small_p && q <= Team::SIZE * kRegRows<Team>) {
                rank_flag = lanes_qr_small<Team::SIZE, kRegRows<Team>>(w.B, q, p, w.rhs, w.vhead, w.tau, small);
                return;
            }
        }
        if constexpr (!is_lane_team<Team>::value) {
            // the CTA bins keep the factor, with Q^T e_k, for later updates
            bool staged = false;
            if constexpr (Team::STAGED) {
                if (p >= 2 * kPanel) {
                    staged = true;
                    rank_flag = qr_solve_staged<Team, T>(team, w.B, q, p, w.rhs, w.vhead, w.tau, small, (T *)w.stage,
                                                         cap.stage_bytes, w.Tst, w.pnb, w.ho, 0);
                }
            }
            if (!staged) {
                rank_flag = qr_factor_team<Team, T>(team, w.B, q, p, w.rhs, w.vhead, w.tau, small, 0);
                single_panels(0);
            }
            // a factor from scratch: factor order = sorted order
            const int me = team.rank();
            for (int i = me; i < q; i += Team::SIZE) {
                w.qte[i] = w.rhs[i];
                w.Ip[i] = i;
            }
            for (int c = me; c < p; c += Team::SIZE) w.Jp[c] = c;
            team.sync();
            back_substitute_blocked(team, w.B, q, p, w.rhs, small);
            fact_valid = true;
            return;
        }
        rank_flag = qr_solve_team<Team, T>(team, w.B, q, p, w.rhs, w.vhead, w.tau, small);
    }

    // Reflectors j0..p-1 factored one at a time: panels of one (global-memory bins)
    __device__ void single_panels(int j0) {
        if constexpr (Team::STAGED) {
            for (int j = j0 + team.rank(); j < p; j += Team::SIZE) {
                w.pnb[j] = 1;
                w.Tst[(int64_t)j * kPanel] = w.tau[j];
            }
            team.sync();
        }
    }

    // factor row of sorted I position i / factor column of sorted J position c
    __device__ __forceinline__ int frow(int i) const {
        if constexpr (is_lane_team<Team>::value) return i;
        else return cap.append ? w.Ip[i] : i;
    }
    __device__ __forceinline__ int fcol(int c) const {
        if constexpr (is_lane_team<Team>::value) return c;
        else return cap.append ? w.Jp[c] : c;
    }

    // rhs <- R^{-1} Q^T rhs with the stored reflectors
    __device__ void apply_qt_solve(T small) {
        if constexpr (is_lane_team<Team>::value) {
            if (p > 2 && p <= cap.small_p && q <= Team::SIZE * kRegRows<Team>) {
                lanes_apply_qt_small<Team::SIZE, kRegRows<Team>>(w.B, q, p, w.rhs, w.vhead, w.tau, small);
                return;
            }
        }
        if constexpr (Team::STAGED) {
            apply_qt_panels<Team, T>(team, w.B, q, p, w.rhs, w.vhead, w.Tst, w.pnb, (T *)w.stage, cap.stage_bytes);
            back_substitute_blocked(team, w.B, q, p, w.rhs, small);
            return;
        }
        if constexpr (is_lane_team<Team>::value) apply_qt_lanes<Team, T>(team, w.B, q, p, w.rhs, w.vhead, w.tau, small);
        else apply_qt_team<Team, T>(team, w.B, q, p, w.rhs, w.vhead, w.tau, small);
    }

    // J for the products with rows of A: as a map in the staging area, or a copy
    // of it there (Js), or J itself.  Synchronises the team.
    __device__ __forceinline__ StageMap map_of_J(const int32_t *&Js) {
        const int me = team.rank();
        Js = w.J;
        StageMap map(nullptr, 0, A.n);
        if constexpr (Team::STAGED) {
            map = stage_map();
            if (map.on()) {
                map.clear(team);
                for (int c = me; c < p; c += Team::SIZE) map.mark(w.J[c]);
                map.finish(team, nullptr, cap.pcap);
            } else if ((size_t)p * sizeof(int32_t) <= (size_t)cap.stage_bytes) {
                int32_t *jc = reinterpret_cast<int32_t *>(w.stage);
                for (int c = me; c < p; c += Team::SIZE) jc[c] = w.J[c];
                Js = jc;
            }
        }
        team.sync();
        return map;
    }

    // sum over the entries e0 .. e0 + len - 1 of A in row order that lie in J,
    // times x; eight lanes per row, four rows per warp (all lanes call)
    __device__ __forceinline__ double row_dot(int64_t e0, int len, const double *v, const StageMap &map,
                                              const int32_t *Js, int &cnt) const {
        const int sub = team.rank() & 7;
        double acc[4] = {0.0, 0.0, 0.0, 0.0};
        int most = len;
#pragma unroll
        for (int o = 16; o >= 8; o >>= 1) most = max(most, __shfl_xor_sync(0xffffffffu, most, o));
        for (int b = 0; b < most; b += 32) {
#pragma unroll
            for (int h = 0; h < 4; ++h) {
                if (b + 8 * h >= most) break;  // the same for the whole warp
                const int e = b + 8 * h + sub;
                if (e < len) {
                    const int32_t col = A.col_idx[e0 + e];
                    int pos;
                    if (Team::STAGED && map.on()) pos = map.find(col);
                    else pos = find_i32(Js, p, col);
                    if (pos >= 0) {
                        acc[h] = fma(A.val[e0 + e], v[pos], acc[h]);
                        ++cnt;
                    }
                }
            }
        }
        double x = acc[0];
        if (most > 16) {
            x += acc[2];
            x += acc[1] + acc[3];
        } else if (most > 8) {
            x += acc[1];
        }
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
        return x;
    }

    // r on the rows of S and, unless `refine`, rho (CTA teams).  The sum of a row
    // is defined on 32 lane chains (entries l, l + 32, ... of the row on lane l)
    // joined by a butterfly over offsets 16, 8, 4, 2, 1, and ||r||^2 as the
    // chains of the rows w, w + 16, ... for w < 16, added in order, for every CTA
    // size.  FP64 additions are what bounds this (a warp instruction takes the
    // SM's FP64 unit 16 cycles however many of its lanes are active), and most rows
    // hold under 16 entries: so eight lanes work on a row, each keeping its
    // four chains (lanes l, l + 8, l + 16, l + 24), the first two levels of the
    // butterfly are additions within a lane, skipped where all four rows of the
    // warp are short (they would add zeros), and the chains of squares run on
    // 16 lanes of one warp, one each, at the end.
    __device__ __forceinline__ void row_sums(bool refine, int &cnt) {
        const int me = team.rank();
        const int32_t *Js;
        const StageMap map = map_of_J(Js);
        const int sub = me & 7;
        constexpr int RW = Team::SIZE / 8;  // rows per pass of the team
        const int passes = (s + RW - 1) / RW;
        for (int t = 0; t < passes; ++t) {
            const int i = t * RW + (me >> 3);
            int32_t row = -1;
            int64_t e0 = 0;
            int len = 0;
            if (i < s) {
                row = w.S[i];
                e0 = A.row_ptr[row];
                len = (int)(A.row_ptr[row + 1] - e0);
            }
            double x = row_dot(e0, len, w.m, map, Js, cnt);
            if (row == k) x -= 1.0;
            if (sub == 0 && i < s) w.r[i] = x;
        }
        team.sync();
        if (!refine) {
            double ss = 0.0;
            if (me < 32) {
                if (me < kVirtualWarps)
                    for (int i = me; i < s; i += kVirtualWarps) ss = fma(w.r[i], w.r[i], ss);
                double tot = __shfl_sync(0xffffffffu, ss, 0);
#pragma unroll
                for (int v = 1; v < kVirtualWarps; ++v) tot += __shfl_sync(0xffffffffu, ss, v);
                ss = tot;
            }
            rho = sqrt(team.bcast(ss, 0));
        }
    }

    // A(I_i, J) x in double, in ascending j (warp bins); *count += its entries
    __device__ __forceinline__ double row_product(const double *x, int i, int *count) const {
        const double *v = w.row_vals() + w.rstart[i];
        double acc = 0.0;
        uint32_t m = w.rmask[i];
        *count += __popc(m);
        for (; m; m &= m - 1u) acc = fma(*v++, x[__ffs(m) - 1], acc);
        return acc;
    }

    // S = I u {k}; r = A(:,J) m - e_k on S in double (Eq. 2.4), row by row: from
    // the rows kept by the solve, in ascending j (the oracle's order), on the warp
    // bins; through the CSR of A, in row_sums' order, on the CTA bins.
    // `refine`: the residual of a refinement step (counted as refinement work).
    __device__ void residual(bool refine = false) {
        const int me = team.rank();
        int pk = lower_bound_i32(w.I, q, k);
        bool has_k = pk < q && w.I[pk] == k;
        s = has_k ? q : q + 1;
        for (int i = me; i < s; i += Team::SIZE) {
            int32_t row;
            if (has_k) row = w.I[i];
            else row = (i < pk) ? w.I[i] : (i == pk ? k : w.I[i - 1]);
            w.S[i] = row;
        }
        double ss = 0.0;
        int cnt = 0;
        (void)ss;
        if constexpr (!is_lane_team<Team>::value) {
            // CTA teams: eight lanes per row, four rows per warp; see row_sums
            row_sums(refine, cnt);
        } else {
            team.sync();
            for (int i = me; i < s; i += Team::SIZE) {
                const bool own = !has_k && i == pk;  // row k, not in I: no entries
                double acc = own ? 0.0 : row_product(w.m, has_k || i < pk ? i : i - 1, &cnt);
                if (w.S[i] == k) acc -= 1.0;
                w.r[i] = acc;
                if (!refine) ss = fma(acc, acc, ss);
            }
        }
        // the refinement step reads r only; its norm is not formed
        if constexpr (is_lane_team<Team>::value) {
            if (!refine) rho = sqrt(team.sum(ss));
        }
        long long nnzJ = team.sum(cnt);
        if (refine) c_ref64 += 2 * nnzJ + 2 * (long long)s;
        else c_res += 2 * nnzJ + 2 * (long long)s;
        team.sync();
    }

    // One step of refinement (FP32_REFINE): r = B m - e in double,
    // m += R^{-1} Q^T (-r) with the factor of the last solve.
    __device__ __forceinline__ void refine_step(T small) {
        const int me = team.rank();
        residual(true);
        int pk = lower_bound_i32(w.I, q, k);
        bool has_k = pk < q && w.I[pk] == k;
        for (int i = me; i < q; i += Team::SIZE) {
            int si = (has_k || i < pk) ? i : i + 1;
            w.rhs[frow(i)] = (T)(-w.r[si]);
        }
        team.sync();
        apply_qt_solve(small);
        for (int c = me; c < p; c += Team::SIZE) w.m[c] += (double)w.rhs[fcol(c)];
        team.sync();
        c_ref += 4LL * q * p + (long long)p * p;
    }

    __device__ __forceinline__ void count_solve(bool append) {
        c_qr += append ? solve_flops(q0, p0, q, p) : solve_flops(0, 0, q, p);
        q0 = q;
        p0 = p;
        c_solves += 1;
        c_pmax = max(c_pmax, p);
        c_qmax = max(c_qmax, q);
    }

    // I = sorted rows of A(:,J) and B = A(I,J) with e_k in rhs, for teams within a warp
    // (|J| <= their lanes: lane c holds column c): each entry is looked up in I once,
    // and the rows that the residuals need are kept beside B (row_vals), instead
    // of walking the rows of A with a search of J per entry: a row holds seven
    // entries of A and two or three of J on a 3-D stencil.  False on overflow.
    __device__ __forceinline__ bool gather_lanes(T *fro2s) {
        const int me = team.rank();
        int len = 0;
        int64_t st = 0;
        if (me < p) {
            st = A.col_ptr[w.J[me]];
            len = counted_entries(A.col_ptr[w.J[me] + 1] - st, cap.scap);
        }
        int tot;
        const int off = team.scan(len, &tot);
        if (tot > cap.scap) return false;
        for (int e = 0; e < len; e += 4) {
            int32_t v[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) v[u] = (e + u < len) ? A.row_idx[st + e + u] : 0;
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (e + u < len) w.buf[off + e + u] = v[u];
        }
        team.sync();
        team_sort_i32(team, w.buf, tot);
        const int nq = team_unique_i32(team, w.buf, tot, w.buf2);
        if (nq > cap.qcap) return false;
        q = nq;
        if ((int64_t)q * p > cap.bcap) return false;
        for (int i = me; i < q; i += Team::SIZE) {
            const int32_t row = w.buf2[i];
            w.I[i] = row;
            w.rhs[i] = row == k ? T(1) : T(0);
            w.rmask[i] = 0u;
        }
        fill_zero(w.B, q * p);
        team.sync();
        uint8_t *pos = reinterpret_cast<uint8_t *>(w.wv);  // of every entry in I (|I| <= 128)
        T fro2 = 0;
        T *Bc = w.B + (int64_t)me * q;
        for (int e = 0; e < len; e += 4) {
            int32_t ri[4];
            T av[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                ri[u] = (e + u < len) ? A.row_idx[st + e + u] : -1;
                av[u] = (e + u < len) ? csc_value<T>(A, st + e + u) : T(0);
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                if (ri[u] >= 0) {
                    const T a = av[u];
                    const int i = find_i32(w.I, q, ri[u]);
                    Bc[i] = a;
                    fro2 += a * a;
                    pos[off + e + u] = (uint8_t)i;
                    atomicOr(&w.rmask[i], 1u << me);
                }
            }
        }
        *fro2s = team.sum(fro2);
        team.sync();
        int base = 0;
        for (int i0 = 0; i0 < q; i0 += Team::SIZE) {
            const int i = i0 + me;
            int part;
            const int at = team.scan(i < q ? __popc(w.rmask[i]) : 0, &part);
            if (i < q) w.rstart[i] = base + at;
            base += part;
        }
        team.sync();
        double *rv = w.row_vals();
        for (int e = 0; e < len; ++e) {
            const int i = pos[off + e];
            rv[w.rstart[i] + __popc(w.rmask[i] & ((1u << me) - 1u))] = A.cval[st + e];
        }
        return true;
    }

    // x[0..len) = 0 (x 16-byte aligned), 16 bytes per store
    __device__ __forceinline__ void fill_zero(T *x, int len) const {
        constexpr int CW = 16 / (int)sizeof(T);
        const int full = len / CW;
        for (int i = team.rank(); i < full; i += Team::SIZE) reinterpret_cast<uint4 *>(x)[i] = make_uint4(0, 0, 0, 0);
        for (int i = full * CW + team.rank(); i < len; i += Team::SIZE) x[i] = T(0);
    }
    // position of row i in I while the staging area holds the map of I (after rows_of_J, in cols_times)
    __device__ __forceinline__ int find_I(int32_t i) const {
        if constexpr (Team::STAGED) {
            const StageMap map = stage_map();
            if (map.on()) return map.find(i);
        }
        return find_i32(w.I, q, i);
    }

    // Solve the LS problem on the current J (Eq. 2.3).  `append`: J extends
    // the previously solved J by Jhat (the paper's QR update; counted as
    // such).  The CTA bins (Caps::append) then update the kept factor instead
    // of refactoring when the last solve left one.
    __device__ bool solve(bool append) {
        const int me = team.rank();
        if constexpr (!is_lane_team<Team>::value) {
            if (cap.append && append && fact_valid) {
                const int st = update_factor();
                if (st == 0) return false;
                if (st > 0) {
                    if (P.precision == RSAI_FP32_REFINE) refine_step(small_last);
                    count_solve(append);
                    return true;
                }
            }
            fact_valid = false;
        }
        T fro2s;
        if constexpr (is_lane_team<Team>::value) {
            if (!gather_lanes(&fro2s)) return false;
        } else {
            if (!rows_of_J()) return false;
            if ((int64_t)q * p > cap.bcap) return false;
            // B = A(I,J), zero-filled
            fill_zero(w.B, q * p);
            for (int i = me; i < q; i += Team::SIZE) w.rhs[i] = (w.I[i] == k) ? T(1) : T(0);
            team.sync();
            T fro2 = 0;
            // column by column: column J[c] of A (CSC, the entries rows_of_J has just
            // read) placed by the position of its rows in I
            for (int c = me; c < p; c += Team::SIZE) {
                const int32_t j = w.J[c];
                const int64_t e0 = A.col_ptr[j], e1 = A.col_ptr[j + 1];
                T *Bc = w.B + (int64_t)c * q;
                for (int64_t e = e0; e < e1; e += 4) {
                    int32_t ri[4];
                    T av[4];
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        ri[u] = (e + u < e1) ? A.row_idx[e + u] : -1;
                        av[u] = (e + u < e1) ? csc_value<T>(A, e + u) : T(0);
                    }
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        if (ri[u] >= 0) {
                            const T a = av[u];
                            Bc[find_I(ri[u])] = a;
                            fro2 += a * a;
                        }
                    }
                }
            }
            fro2s = team.sum(fro2);
        }
        if constexpr (!is_lane_team<Team>::value) fro2_f = fro2s;
        T fro = sqrt(fro2s);
        team.sync();
        const T small = T(q) * T(2.0 * Unit<T>::u) * fro;
        small_last = small;
        rank_flag = 0;
        if (q < p) {  // more unknowns than rows: only possible for singular A
            for (int c = me; c < p; c += Team::SIZE) w.m[c] = 0.0;
            rank_flag = 1;
            team.sync();
        } else {
            qr_solve(small);
            for (int c = me; c < p; c += Team::SIZE) w.m[c] = (double)w.rhs[c];
            team.sync();
            if (P.precision == RSAI_FP32_REFINE) refine_step(small);
        }
        count_solve(append);
        return true;
    }

    // The QR update of Section 3 (CTA bins).  J grew by Jhat (sorted, in
    // w.buf[0..p - p0)) since the last solve, whose factor is kept in factor
    // order: the rows and columns of earlier solves first, in the order in
    // which they entered, the new ones after them (w.Ip / w.Jp give the factor
    // position of each sorted I / J entry, w.qte holds Q^T e_k).  The new rows
    // of I are zero in the old columns, so the old reflectors act on the
    // appended columns only (qr_update_apply); the appended block is then
    // factored below row p0.  Returns 1 when m holds the solution, 0 on
    // overflow, -1 when the caller has to solve from scratch (q < p).
    __device__ int update_factor() {
        const int me = team.rank();
        const int qo = (int)q0, po = (int)p0, nj = p - po;
        fact_valid = false;
        // Jhat and the old sorted I are kept (rows_of_J reuses buf; the
        // residual rewrites S afterwards)
        for (int b = me; b < nj; b += Team::SIZE) w.Jn[b] = w.buf[b];
        for (int i = me; i < qo; i += Team::SIZE) w.S[i] = w.I[i];
        team.sync();
        if (!rows_of_J()) return 0;
        if ((int64_t)q * p > cap.bcap) return 0;
        if (q < p || q > cap.scap || p > cap.scap) return -1;
        // factor rows: old rows keep theirs, new rows follow in ascending order
        int32_t *ipn = w.buf2, *jpn = w.buf;
        int base = 0;
        for (int i0 = 0; i0 < q; i0 += Team::SIZE) {
            const int i = i0 + me;
            const int io = (i < q) ? find_i32(w.S, qo, w.I[i]) : 0;
            const int fnew = (i < q) && (io < 0);
            int tot;
            const int pos = team.scan(fnew, &tot);
            if (i < q) ipn[i] = fnew ? qo + base + pos : w.Ip[io];
            base += tot;
        }
        // factor columns: the old ones keep theirs, Jhat follows in ascending
        // order (an old column is the (c - b)-th of the old sorted J when b
        // entries of Jhat precede it)
        for (int c = me; c < p; c += Team::SIZE) {
            const int b = lower_bound_i32(w.Jn, nj, w.J[c]);
            jpn[c] = (b < nj && w.Jn[b] == w.J[c]) ? po + b : w.Jp[min(max(c - b, 0), po - 1)];
        }
        team.sync();
        for (int i = me; i < q; i += Team::SIZE) w.Ip[i] = ipn[i];
        for (int c = me; c < p; c += Team::SIZE) w.Jp[c] = jpn[c];
        // B: leading dimension q0 -> q in place (column 0 stays).  Old flat
        // index o moves to (o / q0) q + o % q0 >= o, so chunks taken from the
        // top down, each read into registers before any of it is written,
        // never overwrite an entry that is still to be read.
        if (q > qo) {
            constexpr int K = 8;
            constexpr int64_t chunk = (int64_t)K * Team::SIZE;
            for (int64_t hi = (int64_t)qo * po; hi > qo; hi -= chunk) {
                const int64_t lo = max((int64_t)qo, hi - chunk);
                T v[K];
#pragma unroll
                for (int u = 0; u < K; ++u) {
                    const int64_t o = lo + me + (int64_t)u * Team::SIZE;
                    v[u] = (o < hi) ? w.B[o] : T(0);
                }
                team.sync();
#pragma unroll
                for (int u = 0; u < K; ++u) {
                    const int64_t o = lo + me + (int64_t)u * Team::SIZE;
                    if (o < hi) {  // at most bcap elements: 32-bit quotients
                        const unsigned col = (unsigned)o / (unsigned)qo;
                        w.B[(int64_t)col * q + ((unsigned)o - col * (unsigned)qo)] = v[u];
                    }
                }
            }
            team.sync();
            const unsigned nr = (unsigned)(q - qo);
            for (unsigned idx = me; idx < (unsigned)po * nr; idx += Team::SIZE) {
                const unsigned c = idx / nr;
                w.B[(int64_t)c * q + qo + (idx - c * nr)] = T(0);
            }
        }
        for (int64_t idx = (int64_t)po * q + me; idx < (int64_t)p * q; idx += Team::SIZE) w.B[idx] = T(0);
        for (int f = qo + me; f < q; f += Team::SIZE) w.qte[f] = T(0);
        team.sync();
        // the appended columns, placed by the factor row of each entry
        T fro2 = 0;
        for (int b = me; b < nj; b += Team::SIZE) {
            const int32_t j = w.Jn[b];
            T *Bc = w.B + (int64_t)(po + b) * q;
            for (int64_t e = A.col_ptr[j]; e < A.col_ptr[j + 1]; ++e) {
                const T a = csc_value<T>(A, e);
                const int ii = find_I(A.row_idx[e]);
                if (ii >= 0) Bc[w.Ip[ii]] = a;
                fro2 += a * a;
            }
        }
        fro2_f += team.sum(fro2);
        const T small = T(q) * T(2.0 * Unit<T>::u) * sqrt(fro2_f);
        small_last = small;
        // e_k on the new rows: k enters I late when a drop had removed it
        if (me == 0) {
            const int ik = lower_bound_i32(w.I, q, k);
            if (ik < q && w.I[ik] == k && w.Ip[ik] >= qo) w.qte[w.Ip[ik]] = T(1);
        }
        team.sync();
        bool staged = false;
        if constexpr (Team::STAGED) {
            qr_update_apply_staged<Team, T>(team, w.B, q, p, qo, po, w.vhead, w.tau, (T *)w.stage, cap.stage_bytes,
                                            w.Tst, w.pnb, w.ho);
            if (p >= 2 * kPanel) {
                staged = true;
                qr_solve_staged<Team, T>(team, w.B, q, p, w.qte, w.vhead, w.tau, small, (T *)w.stage,
                                         cap.stage_bytes, w.Tst, w.pnb, w.ho, po);
            }
        } else {
            update_reflectors(team, w.B, q, p, qo, po, w.vhead, w.tau, 0, po);
        }
        if (!staged) {
            qr_factor_team<Team, T>(team, w.B, q, p, w.qte, w.vhead, w.tau, small, po);
            single_panels(po);
        }
        int rf = 0;
        for (int j = me; j < p; j += Team::SIZE) rf |= (fabs(w.B[(int64_t)j * q + j]) <= small) ? 1 : 0;
        rank_flag = team.sum(rf) > 0 ? 1 : 0;
        for (int j = me; j < p; j += Team::SIZE) w.rhs[j] = w.qte[j];
        team.sync();
        back_substitute_blocked(team, w.B, q, p, w.rhs, small);
        for (int c = me; c < p; c += Team::SIZE) w.m[c] = (double)w.rhs[w.Jp[c]];
        team.sync();
        fact_valid = true;
        return 1;
    }

    // D = D u (dropped columns of J not yet in D); `kept` marks the columns
    // that stay.  False if D outgrows its capacity.
    template <class Kept> __device__ bool note_dropped(Kept kept) {
        const int me = team.rank();
        int nt = 0;
        for (int c0 = 0; c0 < p; c0 += Team::SIZE) {
            const int c = c0 + me;
            const int f = (c < p) && !kept(c) && find_i32(w.D, nD, w.J[c]) < 0;
            int tot;
            const int pos = team.scan(f, &tot);
            if (f) w.buf2[nt + pos] = w.J[c];
            nt += tot;
        }
        team.sync();
        if (nD + nt > cap.dcap) return false;
        // merge by ranks (both sorted and disjoint) into buf, then back into D
        for (int a = me; a < nD; a += Team::SIZE) w.buf[a + lower_bound_i32(w.buf2, nt, w.D[a])] = w.D[a];
        for (int b = me; b < nt; b += Team::SIZE) w.buf[b + lower_bound_i32(w.D, nD, w.buf2[b])] = w.buf2[b];
        team.sync();
        nD += nt;
        for (int a = me; a < nD; a += Team::SIZE) w.D[a] = w.buf[a];
        team.sync();
        return true;
    }

    // Eq. 4.3: drop |m_j| <= tau, keep at least the largest, re-solve once.
    // Magnitudes are compared as ordered integer keys (exact).
    // Returns 1 if J lost entries (the caller re-solves once), 0 if not, -1
    // if the set of dropped columns outgrows this bin.
    __device__ int drop() {
        if (P.drop_mode == RSAI_DROP_NONE) return 0;
        const int me = team.rank();
        const int blk = P.col_block ? P.col_block[k] : 0;
        const double tau = (P.drop_mode == RSAI_DROP_ADAPTIVE) ? P.eps / ((double)p * P.norm1[blk]) : P.tau_fixed[blk];
        const long long tk = abskey(tau);
        int nkeep = 0;
        long long ba = -1;
        int bi = INT32_MAX;
        for (int c = me; c < p; c += Team::SIZE) {
            long long a = abskey(w.m[c]);
            nkeep += (a > tk);
            if (dom_before(a, c, ba, bi)) { ba = a; bi = c; }
        }
        const int keep_total = team.sum(nkeep);
        if (keep_total == p) return 0;
        if (keep_total == 0) {
            team.argmax(ba, bi);
            if (p == 1) return 0;
            if (!note_dropped([&](int c) { return c == bi; })) return -1;
            int32_t jb = w.J[bi];
            team.sync();
            if (me == 0) w.J[0] = jb;
            p = 1;
            team.sync();
        } else {
            if (!note_dropped([&](int c) { return abskey(w.m[c]) > tk; })) return -1;
            int base = 0;
            for (int c0 = 0; c0 < p; c0 += Team::SIZE) {
                int c = c0 + me;
                int f = (c < p) && (abskey(w.m[c]) > tk);
                int tot;
                int pos = team.scan(f, &tot);
                if (f) w.Jn[base + pos] = w.J[c];
                base += tot;
            }
            team.sync();
            for (int c = me; c < base; c += Team::SIZE) w.J[c] = w.Jn[c];
            p = base;
            team.sync();
        }
        c_drops += 1;
        return 1;
    }

    // Top-c dominant rows of S \ R (Algorithm 1, Eq. 3.2) into w.Rhat; returns
    // their number (0: no candidate left).  |r_i| enters only as ordered
    // integer keys; the tie band needs three double operations per call.
    __device__ int dominant_rows() {
        const int me = team.rank();
        long long rinf = 0;
        for (int i = me; i < s; i += Team::SIZE) rinf = max(rinf, abskey(w.r[i]));
        rinf = team.maxv(rinf);
        const double band = P.tie_band * key_value(rinf);
        const long long bk = abskey(band);
        int ncand = 0;
        for (int i = me; i < s; i += Team::SIZE)
            ncand += (abskey(w.r[i]) > bk) && (find_i32(w.Rset, nR, w.S[i]) < 0);
        ncand = team.sum(ncand);
        if (ncand == 0) return 0;
        const int c = P.c;
        const bool take_all = ncand <= c;
        long long hik = 0, lob = 0;
        if (!take_all) {
            // the c-th element of the (|r| desc, i asc) order: c rounds of argmax,
            // each over the candidates strictly after the previous pick
            long long pa = LLONG_MAX;
            int pi = -1;
            for (int t = 0; t < c; ++t) {
                long long ba = -1;
                int bi = INT32_MAX;
                for (int i = me; i < s; i += Team::SIZE) {
                    long long a = abskey(w.r[i]);
                    int32_t row = w.S[i];
                    if (a > bk && dom_before(pa, pi, a, row) && dom_before(a, row, ba, bi) &&
                        find_i32(w.Rset, nR, row) < 0) {
                        ba = a;
                        bi = row;
                    }
                }
                team.argmax(ba, bi);
                pa = ba;
                pi = bi;
            }
            const double v = key_value(pa);
            hik = abskey(v + band);
            lob = __double_as_longlong(v - band);  // negative bit pattern if v - band < 0
        }
        // selection in index order: all candidates, or (above v + band) +
        // (lowest-index entries within [v - band, v + band] up to c)
        int nabove = 0;
        if (!take_all) {
            for (int i = me; i < s; i += Team::SIZE) {
                long long a = abskey(w.r[i]);
                nabove += (a > bk) && (a > hik) && (find_i32(w.Rset, nR, w.S[i]) < 0);
            }
            nabove = team.sum(nabove);
        }
        const int need = c - nabove;
        int base = 0, tbase = 0;
        for (int i0 = 0; i0 < s; i0 += Team::SIZE) {
            int i = i0 + me;
            int cand = 0, above = 0, tie = 0;
            if (i < s) {
                long long a = abskey(w.r[i]);
                cand = (a > bk) && (find_i32(w.Rset, nR, w.S[i]) < 0);
                if (cand && !take_all) {
                    above = a > hik;
                    tie = (a >= lob) && (a <= hik);
                }
            }
            int ttot;
            int trank = team.scan(tie, &ttot);
            int sel = take_all ? cand : (above || (tie && (tbase + trank) < need));
            int tot;
            int pos = team.scan(sel, &tot);
            if (sel) w.Rhat[base + pos] = w.S[i];
            base += tot;
            tbase += ttot;
        }
        team.sync();
        return base;
    }

    // R = R u Rhat (sorted); false if R outgrows its capacity
    __device__ bool add_to_R(int nh) {
        if (nR + nh > cap.rcap) return false;
        if (team.rank() == 0) {
            for (int t = 0; t < nh; ++t) {
                int32_t x = w.Rhat[t];
                int at = nR + t;
                while (at > 0 && w.Rset[at - 1] > x) { w.Rset[at] = w.Rset[at - 1]; --at; }
                w.Rset[at] = x;
            }
        }
        nR += nh;
        team.sync();
        return true;
    }

    // Jhat = cols(A(Rhat,:)) \ J into w.buf; returns |Jhat| or -1 on overflow.
    // The rows of Rhat are dealt out to the team's ranks, as many passes as
    // |Rhat| (<= c <= 32) needs on a team of 16.  In the global-memory bins a
    // warp takes a row and the columns are collected in the staging area's map.
    __device__ int new_columns(int nh) {
        const int me = team.rank();
        if constexpr (Team::STAGED) {
            const StageMap map = stage_map();
            if (map.on()) {
                map.clear(team);
                int entries = 0;
                for (int t = me >> 5; t < nh; t += Team::SIZE / 32) {
                    const int64_t st = A.row_ptr[w.Rhat[t]];
                    const int len = counted_entries(A.row_ptr[w.Rhat[t] + 1] - st, cap.scap);
                    if ((me & 31) == 0) entries += len;
                    for (int e = me & 31; e < len; e += 32) map.mark(A.col_idx[st + e]);
                }
                entries = team.sum(entries);
                if (entries > cap.scap) return -1;
                for (int c = me; c < p; c += Team::SIZE) map.unmark(w.J[c]);
                // at most `entries` <= scap columns: buf holds them
                return map.finish(team, w.buf, cap.scap);
            }
        }
        int tot = 0;
        for (int t0 = 0; t0 < nh; t0 += Team::SIZE) {
            const int t = t0 + me;
            int len = 0;
            int64_t st = 0;
            if (t < nh) {
                st = A.row_ptr[w.Rhat[t]];
                len = counted_entries(A.row_ptr[w.Rhat[t] + 1] - st, cap.scap);
            }
            int part;
            const int off = tot + team.scan(len, &part);
            if (tot + part > cap.scap) return -1;
            for (int e = 0; e < len; e += 4) {
                int32_t v[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) v[u] = (e + u < len) ? A.col_idx[st + e + u] : 0;
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    if (e + u < len) w.buf[off + e + u] = v[u];
            }
            tot += part;
        }
        team.sync();
        team_sort_i32(team, w.buf, tot);
        int nu = team_unique_i32(team, w.buf, tot, w.buf2);
        int base = 0;
        for (int i0 = 0; i0 < nu; i0 += Team::SIZE) {
            int i = i0 + me;
            int f = (i < nu) && (find_J(w.buf2[i]) < 0);
            int t2;
            int pos = team.scan(f, &t2);
            if (f) w.buf[base + pos] = w.buf2[i];
            base += t2;
        }
        team.sync();
        return base;
    }

    // J = J u Jhat (both sorted, disjoint) by merge ranks
    __device__ bool merge_J(int nj) {
        const int me = team.rank();
        need = p + nj;
        if (need > cap.pcap) return false;
        for (int a = me; a < p; a += Team::SIZE) w.Jn[a + lower_bound_i32(w.buf, nj, w.J[a])] = w.J[a];
        for (int b = me; b < nj; b += Team::SIZE) w.Jn[b + lower_bound_i32(w.J, p, w.buf[b])] = w.buf[b];
        team.sync();
        p += nj;
        for (int a = me; a < p; a += Team::SIZE) w.J[a] = w.Jn[a];
        team.sync();
        return true;
    }

    // algorithmic bytes of columns entering J for the first time: 12 per
    // nonzero + 16 of pointers (a column dropped earlier was charged then)
    __device__ void note_bytes_columns(int from, int count, const int32_t *list) {
        long long b = 0;
        for (int t = from + team.rank(); t < from + count; t += Team::SIZE) {
            int32_t j = list[t];
            if (find_i32(w.D, nD, j) < 0) b += 12 * (A.col_ptr[j + 1] - A.col_ptr[j]) + 16;
        }
        c_bytes += team.sum(b);
    }

    // ---- frozen pattern (refit, backward) ----

    // J = Jk (sorted, length pk): false if it does not fit this bin
    __device__ bool load_pattern(const int32_t *Jk, int pk) {
        p = pk; q = 0; s = 0; nR = 0; l = 0; nD = 0; q0 = 0; p0 = 0; rank_flag = 0; rho = 0.0;
        if constexpr (!is_lane_team<Team>::value) fact_valid = false;
        c_qr = c_res = c_ref = c_ref64 = c_bytes = c_sel = 0;
        c_solves = c_drops = c_pmax = c_qmax = 0;
        if (pk > cap.pcap || pk < 1) return false;
        for (int c = team.rank(); c < pk; c += Team::SIZE) w.J[c] = Jk[c];
        team.sync();
        return true;
    }

    // out[i] = sum_c A(I_i, J_c) zc[c] over the rows of I, in double
    __device__ void rows_times(const double *zc, double *out) {
        if constexpr (is_lane_team<Team>::value) {
            int entries = 0;
            for (int i = team.rank(); i < q; i += Team::SIZE) out[i] = row_product(zc, i, &entries);
            team.sync();
            return;
        }
        const int32_t *Js;
        const StageMap map = map_of_J(Js);
        const int me = team.rank();
        constexpr int RW = Team::SIZE / 8;
        int entries = 0;
        for (int i0 = 0; i0 < q; i0 += RW) {
            const int i = i0 + (me >> 3);
            int64_t e0 = 0;
            int len = 0;
            if (i < q) {
                e0 = A.row_ptr[w.I[i]];
                len = (int)(A.row_ptr[w.I[i] + 1] - e0);
            }
            const double x = row_dot(e0, len, zc, map, Js, entries);
            if ((me & 7) == 0 && i < q) out[i] = x;
        }
        team.sync();
    }

    // out[c] = sum_i A(I_i, J_c) v[i] over the columns of J, in double: a lane per
    // column within a warp, eight lanes per column on a CTA (a thread per row or column
    // searched J and I in global memory, ten dependent loads per entry: with the blocked
    // forward substitution and the long rows of k_adjoint_gather, a batch of 8 with its
    // gradient 167.6 -> 161.2 ms)
    __device__ void cols_times(const double *v, double *out) {
        const int me = team.rank();
        if constexpr (is_lane_team<Team>::value) {
            for (int c = me; c < p; c += Team::SIZE) {
                const int32_t j = w.J[c];
                double acc = 0.0;
                for (int64_t e = A.col_ptr[j]; e < A.col_ptr[j + 1]; ++e)
                    acc = fma(A.cval[e], v[find_i32(w.I, q, A.row_idx[e])], acc);
                out[c] = acc;
            }
        } else {
            if constexpr (Team::STAGED) {
                const StageMap map = stage_map();
                if (map.on()) {
                    map.clear(team);
                    for (int i = me; i < q; i += Team::SIZE) map.mark(w.I[i]);
                    map.finish(team, nullptr, cap.qcap);
                }
            }
            constexpr int CP = Team::SIZE / 8;
            for (int c0 = 0; c0 < p; c0 += CP) {
                const int c = c0 + (me >> 3);
                double acc = 0.0;
                if (c < p) {
                    const int64_t e1 = A.col_ptr[w.J[c] + 1];
                    for (int64_t e = A.col_ptr[w.J[c]] + (me & 7); e < e1; e += 8)
                        acc = fma(A.cval[e], v[find_I(A.row_idx[e])], acc);
                }
#pragma unroll
                for (int o = 4; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
                if ((me & 7) == 0 && c < p) out[c] = acc;
            }
        }
        team.sync();
    }

    // rhs[0..p) <- (R^T R)^{-1} rhs[0..p) with R from the last solve
    __device__ void normal_solve(T small) {
        if constexpr (is_lane_team<Team>::value) {
            triangular_lanes<false>(team, w.B, q, p, w.rhs, small);
            triangular_lanes<true>(team, w.B, q, p, w.rhs, small);
            return;
        }
        forward_substitute_blocked(team, w.B, q, p, w.rhs, small, (T *)w.stage, cap.stage_bytes);
        back_substitute_blocked(team, w.B, q, p, w.rhs, small);
    }

    // Refit: solve on the loaded pattern, then the residual.  Returns false on
    // overflow.
    __device__ bool refit() {
        if (!solve(false)) return false;
        residual();
        return true;
    }

    // Adjoint of the frozen-pattern solve of column k (see rsai_backward):
    //   x = m_k(J_k), r = B x - e_k(I_k), z = (B^T B)^{-1} g (one FP64
    //   refinement step in FP32_REFINE), w = B z;  writes r, w over I_k and
    //   alpha = -z + 2 gr x, x over J_k.
    __device__ bool adjoint(const Frozen &F) {
        const int me = team.rank();
        if (!solve(false)) return false;
        residual();
        const int64_t mo = F.Mcolptr[k];
        for (int c = me; c < p; c += Team::SIZE) w.z[c] = F.grad_M[F.Mcsc_to_csr[mo + c]];
        team.sync();
        const T small = small_last;
        for (int c = me; c < p; c += Team::SIZE) w.rhs[c] = (T)w.z[c];
        team.sync();
        normal_solve(small);
        if (P.precision == RSAI_FP32_REFINE) {
            // one refinement step in double: z = z0 + (R^T R)^{-1} (g - B^T B z0);
            // g stays in z, B z0 goes to wv, z0 and B^T B z0 to buffers that a frozen
            // pass does not use otherwise (the warp bins' rows occupy buf and buf2; there
            // D and R hold at least 2 |J| words)
            double *z0 = reinterpret_cast<double *>(is_lane_team<Team>::value ? w.D : w.buf);
            double *u = reinterpret_cast<double *>(is_lane_team<Team>::value ? w.Rset : w.buf2);
            for (int c = me; c < p; c += Team::SIZE) z0[c] = (double)w.rhs[c];
            team.sync();
            rows_times(z0, w.wv);
            cols_times(w.wv, u);
            for (int c = me; c < p; c += Team::SIZE) w.rhs[c] = (T)(w.z[c] - u[c]);
            team.sync();
            normal_solve(small);
            for (int c = me; c < p; c += Team::SIZE) w.z[c] = z0[c] + (double)w.rhs[c];
            team.sync();
        } else {
            for (int c = me; c < p; c += Team::SIZE) w.z[c] = (double)w.rhs[c];
            team.sync();
        }
        rows_times(w.z, w.wv);
        const double gr = F.grad_rho2 ? F.grad_rho2[k] : 0.0;
        const int64_t qo = F.qoff[k];
        int pk = lower_bound_i32(w.I, q, k);
        bool has_k = pk < q && w.I[pk] == k;
        for (int i = me; i < q; i += Team::SIZE) {
            const int si = (has_k || i < pk) ? i : i + 1;
            F.poolI[qo + i] = w.I[i];
            F.poolR[qo + i] = w.r[si];
            F.poolW[qo + i] = w.wv[i];
        }
        for (int c = me; c < p; c += Team::SIZE) {
            const double x = w.m[c];
            F.alphaM[mo + c] = -w.z[c] + 2.0 * gr * x;
            F.xM[mo + c] = x;
        }
        team.sync();
        return true;
    }

    // First solve, J = {k} (Eq. 2.3 with p = 1): I = rows of A(:,k), which the
    // CSC keeps ascending, and m_kk = a_kk / ||a_k||^2 in double (the closed
    // form of the 1-column LS problem; no sort, tile or QR needed).
    __device__ bool initial_solve() {
        const int me = team.rank();
        const int64_t e0 = A.col_ptr[k];
        const int len = (int)(A.col_ptr[k + 1] - e0);
        if (len > cap.qcap) return false;
        double nn = 0.0;
        int kpos = -1;
        for (int i = me; i < len; i += Team::SIZE) {
            const int32_t r = A.row_idx[e0 + i];
            const double a = A.cval[e0 + i];
            w.I[i] = r;
            if constexpr (is_lane_team<Team>::value) {
                w.rmask[i] = 1u;
                w.rstart[i] = i;
                w.row_vals()[i] = a;
            }
            nn = fma(a, a, nn);
            if (r == k) kpos = i;
        }
        nn = team.sum(nn);
        // a_kk found by its position (an integer reduction), not summed in double
        kpos = team.maxv(kpos);
        const double akk = kpos >= 0 ? A.cval[e0 + kpos] : 0.0;
        q = len;
        if (me == 0) w.m[0] = (nn > 0.0) ? akk / nn : 0.0;
        rank_flag = (nn > 0.0) ? 0 : 1;
        c_qr += solve_flops(0, 0, q, 1);
        q0 = q;
        p0 = 1;
        c_solves += 1;
        c_pmax = max(c_pmax, 1);
        c_qmax = max(c_qmax, q);
        team.sync();
        return true;
    }

    __device__ int run() {
        const int me = team.rank();
        p = 1; q = 0; s = 0; nR = 0; l = 0; nD = 0; q0 = 0; p0 = 0; rank_flag = 0; rho = 0.0;
        if constexpr (!is_lane_team<Team>::value) fact_valid = false;
        c_qr = c_res = c_ref = c_ref64 = c_bytes = c_sel = 0;
        c_solves = c_drops = c_pmax = c_qmax = 0;
        if (me == 0) w.J[0] = k;
        team.sync();
        if (P.init_a) {
            // Algorithm 1 started from the initial pattern of A, solved by the
            // general path below
            long long b = 0;
            const int len = pattern_of_column(team, A.col_ptr, A.row_idx, k, cap.pcap, w.J, &b);
            if (len < 0) {
                need = (int)(A.col_ptr[k + 1] - A.col_ptr[k]);
                return COL_OVERFLOW_J;
            }
            p = len;
            c_bytes += b;
        } else {
            c_bytes += 12 * (A.col_ptr[k + 1] - A.col_ptr[k]) + 16;
        }
        // One solve site: the first pass of every round solves on the new J
        // (appended to the last factor after the first round), the second
        // re-solves after a drop (Eq. 4.3); then the residual (Eq. 2.4).
        bool append = false, first = true;
        for (;;) {
            for (int pass = 0; pass < 2; ++pass) {
                // one call site of solve() (it is large and inlined): the
                // closed form covers the first solve of J = {k} only
                if (first && !P.init_a) {
                    if (!initial_solve()) return COL_OVERFLOW;
                } else if (!solve(append)) {
                    return COL_OVERFLOW;
                }
                first = false;
                append = false;
                if (pass == 1) break;
                const int dr = drop();
                if (dr < 0) return COL_OVERFLOW;
                if (dr == 0) break;
            }
            residual();
            bool grown = false;
            while (!grown && rho > P.eps && l < P.l_max) {
                if (P.spai) {
                    const SpaiPick pk = spai_select(team, A, P.c, P.tie_band, cap.scap, w.S, w.r, s, jset(), w.buf,
                                                    w.buf2, w.sc, w.Rhat);
                    c_bytes += pk.bytes;
                    c_sel += pk.sel;
                    const int na = pk.na;
                    if (na < 0) return COL_OVERFLOW;
                    if (na == 0) break;  // no candidate: nothing can be added later either
                    ++l;
                    note_bytes_columns(0, na, w.buf);
                    if (!merge_J(na)) return COL_OVERFLOW_J;
                    grown = true;
                    continue;
                }
                int nh = dominant_rows();
                if (nh == 0) break;
                if (!add_to_R(nh)) return COL_OVERFLOW;
                {
                    long long b = 0;
                    for (int t = me; t < nh; t += Team::SIZE) b += 4 * (A.row_ptr[w.Rhat[t] + 1] - A.row_ptr[w.Rhat[t]]) + 16;
                    c_bytes += team.sum(b);
                }
                int nj = new_columns(nh);
                if (nj < 0) return COL_OVERFLOW;
                ++l;
                if (nj == 0) continue;  // empty Jhat: back to the loop test (Algorithm 1)
                note_bytes_columns(0, nj, w.buf);
                if (!merge_J(nj)) return COL_OVERFLOW_J;
                grown = true;
            }
            if (!grown) break;
            append = true;
        }
        c_bytes += 36LL * p;
        return COL_DONE;
    }
};

}  // namespace rsai
