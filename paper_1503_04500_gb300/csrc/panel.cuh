// panel.cuh -- blocked (compact-WY) Householder QR for the bins whose workspace
// is in global memory: panels of kPanel columns staged in shared memory,
// factored there, and applied to the trailing columns as I - V T V^T.
//
// Arithmetic.  Every sum keeps one fixed order whatever the layout: a dot
// product over rows is 32 lane chains of fused multiply-adds (rows lane,
// lane + 32, ...) joined by a butterfly (trailing updates), or one chain per
// thread, two rows at a time, joined by a butterfly per warp and added over the
// warps (panel steps).  The kernels below change only where operands live and
// how many instructions carry them.
#pragma once

#include <type_traits>

#include "help.cuh"
#include "team_qr.cuh"

namespace rsai {

// Columns of one compact-WY panel
constexpr int kPanel = 16;

// Head of the panel staging area, in elements of T: the panel's T (kPanel x
// kPanel; the panel factorization keeps V^T V below its diagonal), the CTA
// reduction slots (kPanel per warp) and two kPanel-vectors; the staged panel V
// follows, 16-byte aligned.
template <class Team> constexpr int kStageHead = kPanel * kPanel + (Team::SIZE / 32 + 2) * kPanel;

// Layout of a staged panel of nb columns and qq rows (nb * qq elements): the
// columns go in chunks of kChunk = 16 bytes' worth, chunk c an array [qq][kChunk]
// at c * kChunk * qq, so that one 128-bit access takes kChunk columns of a row
// and neighbouring lanes (rows) touch neighbouring 16-byte words: no bank
// conflicts, a quarter of the loads of a column-major panel in FP32.  Columns
// after the last full chunk are stored one by one, at u * qq.
template <typename T> constexpr int kChunk = 16 / (int)sizeof(T);
template <typename T> struct alignas(16) Chunk { T v[kChunk<T>]; };

template <typename T> __device__ __forceinline__ T &panel_at(T *V, int qq, int nb, int r, int u) {
    constexpr int CW = kChunk<T>;
    return (u | (CW - 1)) < nb ? V[(u & ~(CW - 1)) * qq + r * CW + (u & (CW - 1))] : V[u * qq + r];
}

// Columns c*CW .. c*CW+CW-1 of row r (zero past column nb)
template <bool FULL, typename T>
__device__ __forceinline__ Chunk<T> panel_chunk(const T *V, int qq, int nb, int r, int c) {
    constexpr int CW = kChunk<T>;
    if (FULL || (c + 1) * CW <= nb) return *reinterpret_cast<const Chunk<T> *>(V + c * CW * qq + r * CW);
    Chunk<T> x;
#pragma unroll
    for (int k = 0; k < CW; ++k) x.v[k] = (c * CW + k < nb) ? V[(c * CW + k) * qq + r] : T(0);
    return x;
}
template <bool FULL, typename T>
__device__ __forceinline__ void panel_store_chunk(T *V, int qq, int nb, int r, int c, const Chunk<T> &x) {
    constexpr int CW = kChunk<T>;
    if (FULL || (c + 1) * CW <= nb) {
        *reinterpret_cast<Chunk<T> *>(V + c * CW * qq + r * CW) = x;
    } else {
#pragma unroll
        for (int k = 0; k < CW; ++k)
            if (c * CW + k < nb) V[(c * CW + k) * qq + r] = x.v[k];
    }
}

// Panel of nb columns (src: column-major, ld q, at the panel's first diagonal
// element) into the staging area.  heads != NULL: as explicit reflectors, zeros
// above the diagonal and heads[u] on it.  Two rows per thread in flight (32
// coalesced loads).
template <class Team, typename T>
__device__ __forceinline__ void panel_stage(const Team &team, const T *src, int64_t q, T *V, int qq, int nb,
                                            const T *heads) {
    constexpr int CW = kChunk<T>;
    constexpr int RB = sizeof(T) == 8 ? 1 : 2;
    for (int r0 = team.rank(); r0 < qq; r0 += RB * Team::SIZE) {
        Chunk<T> x[RB][kPanel / CW];
#pragma unroll
        for (int b = 0; b < RB; ++b) {
            const int r = r0 + b * Team::SIZE;
#pragma unroll
            for (int u = 0; u < kPanel; ++u) x[b][u / CW].v[u % CW] = (u < nb && r < qq) ? src[u * q + r] : T(0);
        }
#pragma unroll
        for (int b = 0; b < RB; ++b) {
            const int r = r0 + b * Team::SIZE;
            if (r >= qq) break;
            if (heads && r < kPanel) {
#pragma unroll
                for (int u = 0; u < kPanel; ++u) {
                    if (u > r) x[b][u / CW].v[u % CW] = T(0);
                    else if (u == r && u < nb) x[b][u / CW].v[u % CW] = heads[u];
                }
            }
#pragma unroll
            for (int c = 0; c < kPanel / CW; ++c) panel_store_chunk<false>(V, qq, nb, r, c, x[b][c]);
        }
    }
}

// Two independent FP32 fused multiply-adds in one instruction (each rounded as
// fmaf rounds it): half the issue slots of the same work in scalar form.
typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 pack2(float lo, float hi) {
    f32x2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void unpack2(f32x2 x, float &lo, float &hi) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(x));
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
    f32x2 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}

__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b) {
    f32x2 d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
    f32x2 d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}

// a -= f p and acc += a x + b y, acc += a x, element by element of a chunk (each
// element rounded as the scalar expressions contract: one product, then fused)
__device__ __forceinline__ void chunk_sub(Chunk<float> &a, const Chunk<float> &f, float p) {
    const f32x2 np = pack2(-p, -p);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const f32x2 r = fma2(pack2(f.v[2 * h], f.v[2 * h + 1]), np, pack2(a.v[2 * h], a.v[2 * h + 1]));
        unpack2(r, a.v[2 * h], a.v[2 * h + 1]);
    }
}
__device__ __forceinline__ void chunk_sub(Chunk<double> &a, const Chunk<double> &f, double p) {
#pragma unroll
    for (int k = 0; k < 2; ++k) a.v[k] -= f.v[k] * p;
}
__device__ __forceinline__ void chunk_dot(float *acc, const Chunk<float> &a, float x, const Chunk<float> &b, float y) {
    const f32x2 xx = pack2(x, x), yy = pack2(y, y);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        f32x2 t = mul2(pack2(b.v[2 * h], b.v[2 * h + 1]), yy);
        t = fma2(pack2(a.v[2 * h], a.v[2 * h + 1]), xx, t);
        t = add2(pack2(acc[2 * h], acc[2 * h + 1]), t);
        unpack2(t, acc[2 * h], acc[2 * h + 1]);
    }
}
__device__ __forceinline__ void chunk_dot(float *acc, const Chunk<float> &a, float x) {
    const f32x2 xx = pack2(x, x);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const f32x2 t = fma2(pack2(a.v[2 * h], a.v[2 * h + 1]), xx, pack2(acc[2 * h], acc[2 * h + 1]));
        unpack2(t, acc[2 * h], acc[2 * h + 1]);
    }
}
__device__ __forceinline__ void chunk_dot(double *acc, const Chunk<double> &a, double x, const Chunk<double> &b,
                                          double y) {
#pragma unroll
    for (int k = 0; k < 2; ++k) acc[k] += a.v[k] * x + b.v[k] * y;
}
__device__ __forceinline__ void chunk_dot(double *acc, const Chunk<double> &a, double x) {
#pragma unroll
    for (int k = 0; k < 2; ++k) acc[k] += a.v[k] * x;
}

// Sum of kPanel values over the 32 lanes of a warp by halving exchanges (a
// lane keeps the half of its vector that its partner sends back summed): 16
// shuffles instead of 16 x 5, the same additions as a butterfly over offsets
// 16, 8, 4, 2, 1.  Returns the sum of entry lane >> 1.
template <typename T> __device__ __forceinline__ T warp_reduce_scatter16(T (&v)[kPanel], int lane) {
    static_assert(kPanel == 16, "the exchange pattern below is written for 16 values");
#pragma unroll
    for (int h = 8, o = 16; h >= 1; h >>= 1, o >>= 1) {
        const bool up = (lane & o) != 0;
#pragma unroll
        for (int i = 0; i < h; ++i) {
            const T send = up ? v[i] : v[i + h];
            const T keep = up ? v[i + h] : v[i];
            v[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
        }
    }
    return v[0] + __shfl_xor_sync(0xffffffffu, v[0], 1);
}

// Sums of v[0..kPanel) over the CTA: on return lane l of warp 0 holds the sum of
// entry l % kPanel (other warps: nothing).  One synchronisation inside; the
// caller synchronises before red is written again.
template <class Team, typename T>
__device__ __forceinline__ T team_sum16_warp0(const Team &team, T (&v)[kPanel], T *red) {
    constexpr int NW = Team::SIZE / 32;
    const int me = team.rank(), lane = me & 31;
    const T sv = warp_reduce_scatter16(v, lane);
    if ((lane & 1) == 0) red[(me >> 5) * kPanel + (lane >> 1)] = sv;
    team.sync();
    T a = T(0);
    if (me < 32) {
        const int e = lane & (kPanel - 1);
#pragma unroll
        for (int w = lane >> 4; w < NW; w += 2) a += red[w * kPanel + e];
        a += __shfl_xor_sync(0xffffffffu, a, 16);
    }
    return a;
}

// One Householder step t = tc * CW + TK of the panel factorization: a single
// pass over the rows r >= t applies the reflector of step t - 1 to the columns
// u >= t and forms the dot products of column t with every column of the panel
// (the trailing columns' updates, x.x, and Y(s,t) for the earlier reflectors);
// warp 0 then forms the reflector, the factors f of the next pass and row t.
// Chunks are visited from the one that holds column t (rotated by tc) so that
// every register index is a constant.
template <int TK, bool FULL, class Team, typename T>
__device__ __forceinline__ void panel_step(const Team &team, T *V, int qq, int nb, int tc, T *vhead, T *taus, T *tm,
                                           T *red, T *flag, T *f, T small, int &rank_flag) {
    constexpr int CW = kChunk<T>, NC = kPanel / CW;
    const int me = team.rank();
    const int t = tc * CW + TK;
    const bool upd = t > 0 && flag[0] > T(0);
    T acc[kPanel];
#pragma unroll
    for (int u = 0; u < kPanel; ++u) acc[u] = T(0);
    // two rows per thread and iteration: their products are added to a chain together
    for (int ra = t + me; ra < qq; ra += 2 * Team::SIZE) {
        const int rb = ra + Team::SIZE;
        const bool two = rb < qq;
        T pa = T(0), pb = T(0);  // column t - 1
        if (upd) {
            pa = panel_at(V, qq, FULL ? kPanel : nb, ra, t - 1);
            if (two) pb = panel_at(V, qq, FULL ? kPanel : nb, rb, t - 1);
        }
        T xa = T(0), xb = T(0);  // column t
#pragma unroll
        for (int j = 0; j < NC; ++j) {
            const int c = (tc + j) & (NC - 1);
            if (!FULL && c * CW >= nb) continue;
            Chunk<T> a = panel_chunk<FULL>(V, qq, nb, ra, c), b = a;
            if (two) b = panel_chunk<FULL>(V, qq, nb, rb, c);
            if (upd && (j == 0 || c > tc)) {
                Chunk<T> fc = *reinterpret_cast<const Chunk<T> *>(f + c * CW);
                const Chunk<T> a0 = a, b0 = b;
                chunk_sub(a, fc, pa);
                chunk_sub(b, fc, pb);
                if (j == 0) {  // the columns before t are finished
#pragma unroll
                    for (int k = 0; k < TK; ++k) {
                        a.v[k] = a0.v[k];
                        b.v[k] = b0.v[k];
                    }
                }
                panel_store_chunk<FULL>(V, qq, nb, ra, c, a);
                if (two) panel_store_chunk<FULL>(V, qq, nb, rb, c, b);
            }
            if (j == 0) {
                xa = a.v[TK];
                xb = b.v[TK];
            }
            if (two) chunk_dot(acc + j * CW, a, xa, b, xb);
            else chunk_dot(acc + j * CW, a, xa);
        }
    }
    const T s = team_sum16_warp0(team, acc, red);
    if (me < 32) {
        // lane e (and e + 16) holds the dot product of column t with column u
        const int e = me & (kPanel - 1);
        const int u = ((e / CW + tc) & (NC - 1)) * CW + e % CW;
        const T sigma = __shfl_sync(0xffffffffu, s, TK);
        const T x0 = panel_at(V, qq, nb, t, t);
        const T cu = u < nb ? panel_at(V, qq, nb, t, u) : T(0);
        T alpha, v0, two_over;
        reflector(sigma, x0, alpha, v0, two_over);
        __syncwarp();
        if (me < kPanel) {
            if (u == t) {
                tm[t * kPanel + t] = two_over;
                flag[0] = two_over;
                vhead[t] = v0;
                taus[t] = two_over;
                panel_at(V, qq, nb, t, t) = alpha;
            } else if (u < nb) {
                // v_t differs from x only in its head: v_t.c = c.x + (v0 - x0) c_t
                const T d = s + (v0 - x0) * cu;
                if (u > t) {
                    const T fu = d * two_over;
                    f[u] = fu;
                    if (two_over > T(0)) panel_at(V, qq, nb, t, u) = cu - fu * v0;
                } else {
                    tm[t * kPanel + u] = d;  // Y(s,t) for the earlier reflector s = u
                }
            }
        }
        rank_flag |= abs_at_most(alpha, small) ? 1 : 0;
    }
    team.sync();
}

// Householder QR of the staged panel V (rows 0..qq-1, nb <= kPanel columns) with
// the T of its compact-WY form; one pass over the panel and two CTA
// synchronisations per column.  The FP64 square root and division of a step
// run on warp 0 only.  Y(s,t) = v_s.v_t is kept below the diagonal of tm and
// tau_t on it; one warp then forms T(t,t) = tau_t and
// T(s,t) = -tau_t sum_{s <= s2 < t} T(s,s2) Y(s2,t) above it, while the other
// warps write the panel back to B (src, ld q).  Leaves V as explicit reflectors
// (zeros above the diagonal, heads on it), vhead[t] = v0, taus[t] = 2 / v^T v.
// The rank flag is valid on warp 0.
template <class Team, typename T>
__device__ __forceinline__ void panel_factor(const Team &team, T *V, int qq, int nb, T *src, int64_t q, T *vhead,
                                             T *taus, T *tm, T *red, T *flag, T *f, T small, int &rank_flag) {
    constexpr int CW = kChunk<T>;
    const int me = team.rank();
    if (me < kPanel) f[me] = T(0);
    auto steps = [&](auto full) {
        constexpr bool FULL = decltype(full)::value;
        for (int tc = 0; tc * CW < nb; ++tc) {
            panel_step<0, FULL>(team, V, qq, nb, tc, vhead, taus, tm, red, flag, f, small, rank_flag);
            if (FULL || tc * CW + 1 < nb)
                panel_step<1, FULL>(team, V, qq, nb, tc, vhead, taus, tm, red, flag, f, small, rank_flag);
            if constexpr (CW == 4) {
                if (FULL || tc * CW + 2 < nb)
                    panel_step<2, FULL>(team, V, qq, nb, tc, vhead, taus, tm, red, flag, f, small, rank_flag);
                if (FULL || tc * CW + 3 < nb)
                    panel_step<3, FULL>(team, V, qq, nb, tc, vhead, taus, tm, red, flag, f, small, rank_flag);
            }
        }
    };
    if (nb == kPanel) steps(std::true_type{});
    else steps(std::false_type{});
    // T from Y and tau: lane s of warp 0 holds row s of T
    if (me < 32) {
        const int sr = me;
        T trow[kPanel];
#pragma unroll
        for (int t = 0; t < kPanel; ++t) {
            trow[t] = T(0);
            if (t < nb) {
                const T tau = tm[t * kPanel + t];
                T a = T(0);
#pragma unroll
                for (int s2 = 0; s2 < t; ++s2)
                    if (s2 >= sr) a += trow[s2] * tm[t * kPanel + s2];
                if (sr < t) trow[t] = -tau * a;
                else if (sr == t) trow[t] = tau;
            }
        }
        if (sr < nb) {
#pragma unroll
            for (int t = 0; t < kPanel; ++t)
                if (t > sr && t < nb) tm[sr * kPanel + t] = trow[t];
        }
    }
    // R entries and reflector tails to B; then the explicit head of V (each row by its own thread)
    for (int r = me; r < qq; r += Team::SIZE) {
        Chunk<T> x[kPanel / CW];
#pragma unroll
        for (int c = 0; c < kPanel / CW; ++c) x[c] = panel_chunk<false>(V, qq, nb, r, c);
#pragma unroll
        for (int u = 0; u < kPanel; ++u)
            if (u < nb) src[u * q + r] = x[u / CW].v[u % CW];
        if (r < nb) {
#pragma unroll
            for (int u = 0; u < kPanel; ++u) {
                if (u > r) x[u / CW].v[u % CW] = T(0);
                else if (u == r) x[u / CW].v[u % CW] = vhead[u];
            }
#pragma unroll
            for (int c = 0; c < kPanel / CW; ++c) panel_store_chunk<false>(V, qq, nb, r, c, x[c]);
        }
    }
    team.sync();
}

__device__ __forceinline__ void prefetch_l2(const void *p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }

// Passes between the loads of C and their prefetch to L2 in wy_apply_cols.  152
// columns of M have 365 MB of trailing matrices at |I| = 2000, |J| = 300, so
// the first read of a column misses L2: QR of 152 matrices 2800 x 350, 16.8M
// cycles without the prefetch, 12.4M with 6 passes, 12.5M with 12; where
// everything fits L2 it costs 2 %.  Prefetching the second read, which hits, too:
// 13.6M.
constexpr int kAhead = 6;

// C <- C - V (T^T (V^T C)) for KC columns tc[0..KC) (rows 0..qq-1 of each;
// has[x] = false: the column repeats tc[0] and is not stored) on one warp,
// lanes over rows.  Each chain W(u, c) = sum_r V(r,u) C(r,c) runs over the rows
// lane, lane + 32, ... of its lane; the entries of the rows D passes ahead are
// loaded while a pass is computed, so that the loads of C (global memory, L2)
// overlap the arithmetic.  In FP32 the products go two at a time: W pairs
// two reflectors per column, the update pairs two columns.
// A panel of fewer columns (all that fit the staging area of a column of thousands of
// rows) skips in FP64 the chunks past its last: multiplied as zeros they were three quarters
// of the FP64 work of a panel of four (|I| up to 5710: global bin 2387 -> 1686 ms).  In FP32,
// where most such panels are the last ones of short factors, the tests cost more than the
// products (n = 5000 power law, rebuild 132.7 ms without, 135.6 with them).
template <int KC, int D, bool FULL, typename T>
__device__ __forceinline__ void wy_apply_cols(const T *V, int qq, int nb, const T *tm, T *const (&tc)[KC],
                                              const bool (&has)[KC], int lane) {
    constexpr int CW = kChunk<T>, NC = kPanel / CW;
    constexpr bool F32 = sizeof(T) == 4, P2 = F32 && KC >= 2;
    const int full = qq >> 5;  // passes in which every lane has a row
    T cb[D][KC];
    auto load = [&](T (&c)[KC], int r) {
#pragma unroll
        for (int x = 0; x < KC; ++x) c[x] = tc[x][r];
    };
    // f(r, row r of C) over all rows, the loads D passes ahead (the first ones in cb)
    auto stream = [&](auto ahead, auto f) {
        int r = lane, k = 0;
        for (; k + 2 * D <= full; k += D) {
#pragma unroll
            for (int y = 0; y < D; ++y, r += 32) {
                T cur[KC];
#pragma unroll
                for (int x = 0; x < KC; ++x) cur[x] = cb[y][x];
                load(cb[y], r + 32 * D);
                ahead(r + 32 * D);
                f(r, cur);
            }
        }
        if (k + D <= full) {
#pragma unroll
            for (int y = 0; y < D; ++y, r += 32) f(r, cb[y]);
            k += D;
        }
        for (; r < qq; r += 32) {
            T cur[KC];
            load(cur, r);
            f(r, cur);
        }
    };
    auto first = [&] {
        if (full >= D) {
#pragma unroll
            for (int y = 0; y < D; ++y) load(cb[y], lane + 32 * y);
        }
    };
    T nw[KC][kPanel];  // W, then -T^T W
    // W = V^T C
    first();
    {
        f32x2 w2[F32 ? KC : 1][F32 ? kPanel / 2 : 1];
#pragma unroll
        for (int x = 0; x < KC; ++x) {
#pragma unroll
            for (int u = 0; u < kPanel; ++u) {
                if constexpr (F32) w2[x][u / 2] = 0ull;
                else nw[x][u] = T(0);
            }
        }
        stream(
            [&](int r) {
                if (r + 32 * kAhead < qq) {
#pragma unroll
                    for (int x = 0; x < KC; ++x) prefetch_l2(tc[x] + r + 32 * kAhead);
                }
            },
            [&](int r, const T (&cur)[KC]) {
                if constexpr (F32) {
                    f32x2 cc[KC];
#pragma unroll
                    for (int x = 0; x < KC; ++x) cc[x] = pack2(cur[x], cur[x]);
#pragma unroll
                    for (int c = 0; c < NC; ++c) {
                        const Chunk<T> v = panel_chunk<FULL>(V, qq, nb, r, c);
                        const f32x2 v01 = pack2(v.v[0], v.v[1]), v23 = pack2(v.v[2], v.v[3]);
#pragma unroll
                        for (int x = 0; x < KC; ++x) {
                            w2[x][2 * c] = fma2(v01, cc[x], w2[x][2 * c]);
                            w2[x][2 * c + 1] = fma2(v23, cc[x], w2[x][2 * c + 1]);
                        }
                    }
                } else {
#pragma unroll
                    for (int c = 0; c < NC; ++c) {
                        if (!FULL && c * CW >= nb) break;
                        const Chunk<T> v = panel_chunk<FULL>(V, qq, nb, r, c);
#pragma unroll
                        for (int k = 0; k < CW; ++k)
#pragma unroll
                            for (int x = 0; x < KC; ++x) nw[x][c * CW + k] += v.v[k] * cur[x];
                    }
                }
            });
        if constexpr (F32) {
#pragma unroll
            for (int x = 0; x < KC; ++x)
#pragma unroll
                for (int u = 0; u < kPanel / 2; ++u) unpack2(w2[x][u], nw[x][2 * u], nw[x][2 * u + 1]);
        }
    }
    first();  // of the second pass, in flight during the reduction
    // totals: lane l keeps entry u = l >> 1, of column 2g + (l & 1) in sel[g];
    // then -T^T W, one entry per lane and group, and the broadcast to every lane
    {
        constexpr int G = (KC + 1) / 2;
        const int u = lane >> 1, par = lane & 1;
        T sel[G], acc[G];
#pragma unroll
        for (int x = 0; x < KC; ++x) {
            const T tot = warp_reduce_scatter16(nw[x], lane);
            if (x % 2 == 0) sel[x / 2] = tot;
            else sel[x / 2] = par ? tot : sel[x / 2];
        }
#pragma unroll
        for (int g = 0; g < G; ++g) acc[g] = T(0);
#pragma unroll
        for (int s = 0; s < kPanel; ++s) {
            const T ts = tm[s * kPanel + u];
#pragma unroll
            for (int g = 0; g < G; ++g) {
                const T ws = __shfl_sync(0xffffffffu, sel[g], 2 * s + (KC > 1 ? par : 0));
                if (s <= u && u < nb) acc[g] += ts * ws;
            }
        }
#pragma unroll
        for (int g = 0; g < G; ++g) acc[g] = -acc[g];
#pragma unroll
        for (int x = 0; x < KC; ++x)
#pragma unroll
            for (int v = 0; v < kPanel; ++v) nw[x][v] = __shfl_sync(0xffffffffu, acc[x / 2], 2 * v + (x & 1));
    }
    // C <- C + V (-T^T W)
    f32x2 n2[P2 ? KC / 2 : 1][P2 ? kPanel : 1];
    if constexpr (P2) {
#pragma unroll
        for (int g = 0; g < KC / 2; ++g)
#pragma unroll
            for (int u = 0; u < kPanel; ++u) n2[g][u] = pack2(nw[2 * g][u], nw[2 * g + 1][u]);
    }
    stream([](int) {},
           [&](int r, const T (&c0)[KC]) {
               T cur[KC];
#pragma unroll
               for (int x = 0; x < KC; ++x) cur[x] = c0[x];
               if constexpr (P2) {
                   f32x2 a2[KC / 2];
#pragma unroll
                   for (int g = 0; g < KC / 2; ++g) a2[g] = pack2(cur[2 * g], cur[2 * g + 1]);
#pragma unroll
                   for (int c = 0; c < NC; ++c) {
                       const Chunk<T> v = panel_chunk<FULL>(V, qq, nb, r, c);
#pragma unroll
                       for (int k = 0; k < CW; ++k) {
                           const f32x2 vv = pack2(v.v[k], v.v[k]);
#pragma unroll
                           for (int g = 0; g < KC / 2; ++g) a2[g] = fma2(vv, n2[g][c * CW + k], a2[g]);
                       }
                   }
#pragma unroll
                   for (int g = 0; g < KC / 2; ++g) unpack2(a2[g], cur[2 * g], cur[2 * g + 1]);
               } else {
#pragma unroll
                   for (int c = 0; c < NC; ++c) {
                       if (!FULL && !F32 && c * CW >= nb) break;
                       const Chunk<T> v = panel_chunk<FULL>(V, qq, nb, r, c);
#pragma unroll
                       for (int k = 0; k < CW; ++k)
#pragma unroll
                           for (int x = 0; x < KC; ++x) cur[x] += v.v[k] * nw[x][c * CW + k];
                   }
               }
#pragma unroll
               for (int x = 0; x < KC; ++x)
                   if (has[x]) tc[x][r] = cur[x];
           });
}

// Columns c in [c_lo, c_hi] of B (ld q; c == p stands for rhs), rows
// j0..j0+qq-1: C <- C - V (T^T (V^T C)), V staged.  Each warp takes kCols
// columns at a time, fewer once the columns that are left would leave warps
// idle (a reflector value read from shared memory then serves fewer columns,
// but no warp waits for another's extra columns).  Ends with a team
// synchronisation.
template <bool FULL, int KC, int D, class Team, typename T>
__device__ __forceinline__ void wy_apply_group(const Team &team, const T *V, int qq, int nb, const T *tm, T *B, int q,
                                               int p, T *rhs, int j0, int c_lo, int c_hi) {
    const int lane = team.rank() & 31, wid = team.rank() >> 5;
    const int c0 = c_lo + wid * KC;
    if (c0 > c_hi) return;
    T *tc[KC];
    bool has[KC];
#pragma unroll
    for (int x = 0; x < KC; ++x) {
        has[x] = c0 + x <= c_hi;
        const int c = has[x] ? c0 + x : c0;
        tc[x] = (c < p ? B + (int64_t)c * q : rhs) + j0;
    }
    wy_apply_cols<KC, D, FULL>(V, qq, nb, tm, tc, has, lane);
}

template <bool FULL, class Team, typename T>
__device__ __noinline__ void wy_apply(Team team, const T *V, int qq, int nb, const T *tm, T *B, int q, int p, T *rhs,
                                      int j0, int c_lo, int c_hi) {
    constexpr int NW = Team::SIZE / 32;
    constexpr int kCols = sizeof(T) == 8 ? 2 : 4;  // W of kCols x kPanel values stays in registers
    int c = c_lo;
    while (c <= c_hi) {
        const int left = c_hi - c + 1;
        if (kCols == 4 && left > 2 * NW) {
            wy_apply_group<FULL, kCols, 2>(team, V, qq, nb, tm, B, q, p, rhs, j0, c, c_hi);
            c += kCols * NW;
        } else if (left > NW) {
            wy_apply_group<FULL, 2, 2>(team, V, qq, nb, tm, B, q, p, rhs, j0, c, c_hi);
            c += 2 * NW;
        } else {
            wy_apply_group<FULL, 1, 4>(team, V, qq, nb, tm, B, q, p, rhs, j0, c, c_hi);
            c += NW;
        }
    }
    team.sync();
}

template <class Team, typename T>
__device__ __forceinline__ void wy_apply_any(const Team &team, const T *V, int qq, int nb, const T *tm, T *B, int q,
                                             int p, T *rhs, int j0, int c_lo, int c_hi) {
    if (nb == kPanel) wy_apply<true, Team, T>(team, V, qq, nb, tm, B, q, p, rhs, j0, c_lo, c_hi);
    else wy_apply<false, Team, T>(team, V, qq, nb, tm, B, q, p, rhs, j0, c_lo, c_hi);
}

// What a CTA of the global bin needs to share its trailing updates
struct HelpOwner {
    HelpBoard board;
    int slot;        // -1: does not share
    uint32_t epoch;  // of the last published task
    int32_t *err;    // the launch's error word
};

// T of a panel (column t at tcol[t * kPanel]) into tm[s * kPanel + t]
template <class Team, typename T>
__device__ __forceinline__ void load_T(const Team &team, const T *tcol, int nb, T *tm) {
    for (int e = team.rank(); e < kPanel * kPanel; e += Team::SIZE) {
        const int s = e / kPanel, t = e - s * kPanel;
        tm[e] = (t < nb && s <= t) ? tcol[t * kPanel + s] : T(0);
    }
}

// Columns per group of a shared update: a round of the CTA's warps at two (FP64:
// one) columns each, about as long as staging the panel takes a helper ten times
template <class Team, typename T> constexpr int kHelpGroup = Team::SIZE / 32 * (sizeof(T) == 8 ? 1 : 2);

// wy_apply, shared with idle CTAs when there are any (`idle`, as seen by the
// whole team) and at least three groups.  V and T are staged; vhead, tcol: the
// panel's heads and T in the workspace.
template <class Team, typename T>
__device__ __noinline__ void wy_apply_shared(Team team, HelpOwner *ho, bool idle, const T *V, int qq, int nb,
                                             const T *tm, T *B, int q, int p, T *rhs, int j0, int c_lo, int c_hi,
                                             const T *vhead, const T *tcol) {
    constexpr int kGroup = kHelpGroup<Team, T>;
    const int groups = (c_hi - c_lo + kGroup) / kGroup;
    if (!idle || groups < 3 || ho->slot < 0) {
        wy_apply_any(team, V, qq, nb, tm, B, q, p, rhs, j0, c_lo, c_hi);
        return;
    }
    __shared__ int claimed;
    HelpBoard &b = ho->board;
    const int slot = ho->slot;
    const uint32_t epoch = ho->epoch + 1;
    team.sync();  // the panel, its heads and T are written
    if (team.rank() == 0) {
        b.task[slot] = HelpTask{B + (int64_t)j0 * q + j0, vhead, tcol, B, rhs, q, p, qq, nb, j0, c_lo, c_hi, kGroup};
        b.done[slot] = 0u;
        __threadfence();
        atomicExch(&b.word[slot], (unsigned long long)epoch << 32 | (unsigned long long)groups << 16);
    }
    int mine = 0;
    for (;;) {
        if (team.rank() == 0) claimed = help_claim(&b.word[slot], epoch);
        team.sync();
        const int g = claimed;
        team.sync();
        if (g < 0) break;
        ++mine;
        const int c0 = c_lo + g * kGroup;
        wy_apply_any(team, V, qq, nb, tm, B, q, p, rhs, j0, c0, min(c_hi, c0 + kGroup - 1));
    }
    // groups that helpers have claimed
    if (team.rank() == 0) {
        int ok = 1;
        for (unsigned polls = 0; help_load(&b.done[slot]) != (uint32_t)(groups - mine); ++polls)
            if (polls >= kHelpPolls) {
                set_error(ho->err, RSAI_ERR_TIMEOUT);
                ok = 0;
                break;
            }
        __threadfence();
        claimed = ok;
    }
    team.sync();
    ho->epoch = epoch;
    if (!claimed) ho->slot = -1;
    team.sync();
}

// A CTA without a column: groups of other CTAs' updates until all `total`
// columns of the bin are finished.
template <class Team, typename T>
__device__ __noinline__ void help_others(Team team, const HelpBoard &b, uint32_t total, T *stage) {
    __shared__ int pick, claimed, have_slot;
    __shared__ uint32_t have_epoch;
    const int me = team.rank();
    T *tm = stage;
    T *V = stage + kStageHead<Team>;
    if (me == 0) {
        atomicAdd(b.idle, 1u);
        have_slot = -1;
    }
    for (unsigned polls = 0; polls < kHelpPolls; ++polls) {
        // the open task with the most groups left (ties: spread over the helpers)
        int key = -1;
        uint32_t epoch = 0;
        const int slot = me < b.slots ? (me + blockIdx.x) % b.slots : -1;
        if (slot >= 0) {
            const unsigned long long w = help_load(&b.word[slot]);
            const int left = help_groups(w) - help_next(w);
            if (left > 0) key = left * 1024 + me;
            epoch = help_epoch(w);
        }
        const int best = team.maxv(key);
        if (best < 0) {
            if (me == 0) {
                pick = help_load(b.cols_done) >= total ? 1 : 0;
                if (!pick) __nanosleep(400);
            }
            team.sync();
            const bool stop = pick != 0;
            team.sync();
            if (stop) break;
            continue;
        }
        if (key == best) {
            pick = slot;
            const int g = help_claim(&b.word[slot], epoch);
            claimed = g;
            if (g >= 0 && (have_slot != slot || have_epoch != epoch)) {
                have_slot = slot;
                have_epoch = epoch;
                claimed = g | 1 << 20;  // stage the panel first
            }
        }
        team.sync();
        const int got = claimed, sl = pick;
        team.sync();
        if (got < 0) continue;
        polls = 0;
        const int g = got & 0xfffff;
        const HelpTask *tk = &b.task[sl];
        const int q = __ldcg(&tk->q), p = __ldcg(&tk->p), qq = __ldcg(&tk->qq), nb = __ldcg(&tk->nb);
        const int j0 = __ldcg(&tk->j0), c_lo = __ldcg(&tk->c_lo), c_hi = __ldcg(&tk->c_hi), group = __ldcg(&tk->group);
        T *B = (T *)__ldcg((const unsigned long long *)&tk->B);
        T *rhs = (T *)__ldcg((const unsigned long long *)&tk->rhs);
        if (got >> 20) {
            panel_stage(team, (const T *)__ldcg((const unsigned long long *)&tk->src), (int64_t)q, V, qq, nb,
                        (const T *)__ldcg((const unsigned long long *)&tk->heads));
            load_T(team, (const T *)__ldcg((const unsigned long long *)&tk->tcol), nb, tm);
            team.sync();
        }
        const int c0 = c_lo + g * group;
        wy_apply_any(team, V, qq, nb, tm, B, q, p, rhs, j0, c0, min(c_hi, c0 + group - 1));
        if (me == 0) {
            __threadfence();
            atomicAdd(&b.done[sl], 1u);
        }
    }
}

// rhs <- Q^T rhs with the reflectors in the panels they were factored in
// (pnb, Tst): per panel w = V^T rhs (one CTA reduction), y = T^T w, and
// rhs <- rhs - V y, with V = the explicit reflectors (vhead on the diagonal,
// the tails of B below it).  A panel is taken in sub-panels of as many
// reflectors as the staging area holds (the diagonal blocks of its T).  Both
// passes run over a thread's own rows, so the staging area is the thread's
// private copy of them (no synchronisation); when fewer than two reflectors
// fit, or one is left, the second pass reads the slab again.
template <class Team, typename T>
__device__ __noinline__ void apply_qt_panels(Team team, const T *B, int q, int p, T *rhs, const T *vhead,
                                             const T *Tst, const int32_t *pnb, T *stage, int stage_bytes) {
    constexpr int CW = kChunk<T>, NC = kPanel / CW;
    const int me = team.rank();
    T *red = stage + kPanel * kPanel, *y = red + (Team::SIZE / 32 + 1) * kPanel;
    T *V = stage + kStageHead<Team>;
    const int64_t velems = (int64_t)stage_bytes / (int64_t)sizeof(T) - kStageHead<Team>;
    for (int jp = 0; jp < p;) {
        const int nbp = pnb[jp];
        for (int js = 0; js < nbp;) {
            const int j0 = jp + js;
            const int qq = q - j0;
            const int64_t fit = velems / (int64_t)max(qq, 1);
            const bool staged = nbp - js > 1 && fit >= 2;
            const int nb = staged ? (int)min((int64_t)(nbp - js), fit) : nbp - js;
            const T *src = B + (int64_t)j0 * q + j0;
            // column e of T, for lane e of warp 0 (loaded before it is needed)
            T tcol[kPanel];
#pragma unroll
            for (int s = 0; s < kPanel; ++s)
                tcol[s] = (me < nb && s <= me) ? Tst[(int64_t)(j0 + me) * kPanel + js + s] : T(0);
            T acc[kPanel];
#pragma unroll
            for (int u = 0; u < kPanel; ++u) acc[u] = T(0);
            for (int r = me; r < qq; r += Team::SIZE) {
                Chunk<T> v[NC];
#pragma unroll
                for (int u = 0; u < kPanel; ++u) v[u / CW].v[u % CW] = (u < nb) ? src[(int64_t)u * q + r] : T(0);
                const T x = rhs[j0 + r];
                if (r < kPanel) {
#pragma unroll
                    for (int u = 0; u < kPanel; ++u) {
                        if (u > r) v[u / CW].v[u % CW] = T(0);
                        else if (u == r && u < nb) v[u / CW].v[u % CW] = vhead[j0 + u];
                    }
                }
                if (staged) {
#pragma unroll
                    for (int c = 0; c < NC; ++c) panel_store_chunk<false>(V, qq, nb, r, c, v[c]);
                }
#pragma unroll
                for (int u = 0; u < kPanel; ++u)
                    if (u < nb) acc[u] += v[u / CW].v[u % CW] * x;
            }
            const T s = team_sum16_warp0(team, acc, red);
            if (me < 32) {
                T a = T(0);
#pragma unroll
                for (int s2 = 0; s2 < kPanel; ++s2) {
                    const T ws = __shfl_sync(0xffffffffu, s, s2);
                    if (s2 <= me) a += tcol[s2] * ws;
                }
                if (me < kPanel) y[me] = me < nb ? a : T(0);
            }
            team.sync();
            for (int r = me; r < qq; r += Team::SIZE) {
                T a = rhs[j0 + r];
                if (staged) {
#pragma unroll
                    for (int c = 0; c < NC; ++c) {
                        const Chunk<T> v = panel_chunk<false>(V, qq, nb, r, c);
#pragma unroll
                        for (int k = 0; k < CW; ++k)
                            if (c * CW + k < nb) a -= v.v[k] * y[c * CW + k];
                    }
                } else {
#pragma unroll
                    for (int u = 0; u < kPanel; ++u) {
                        if (u < nb) {
                            const T v = (r > u) ? src[(int64_t)u * q + r] : ((r == u) ? vhead[j0 + u] : T(0));
                            a -= v * y[u];
                        }
                    }
                }
                rhs[j0 + r] = a;
            }
            team.sync();
            js += nb;
        }
        jp += nbp;
    }
}

// Blocked Householder QR (compact WY).  Panels of nb <= kPanel columns (nb
// chosen so that rows j0..q of the panel fit the shared-memory staging area) are
// copied there, factored with their T (panel_factor), written back, and every
// trailing column and the right-hand side get
//   C <- C - V (T^T (V^T C)),  H_1...H_nb = I - V T V^T,
// so the trailing matrix in global memory is streamed once per panel instead
// of once per reflector (by this CTA and, when others have run out of columns,
// by them: wy_apply_shared).  Each panel's size and T are kept (pnb, Tst) for
// the QR update and the refinement.  A panel that does not fit four columns
// falls back to single Householder steps (panels of one).  j_start > 0 factors
// only columns j_start..p-1 (the columns appended to a factor whose first
// j_start columns are done, Section 3).  Leaves Q^T rhs in rhs; the rank flag is
// valid on warp 0.
template <class Team, typename T>
__device__ __noinline__ int qr_solve_staged(Team team, T *B, int q, int p, T *rhs, T *vhead, T *taus, T small,
                                            T *stage, int stage_bytes, T *Tst, int32_t *pnb, HelpOwner *ho,
                                            int j_start) {
    const int me = team.rank();
    constexpr int NW = Team::SIZE / 32;
    T *tm = stage;                                  // kPanel x kPanel
    T *red = stage + kPanel * kPanel;               // reduction slots
    T *flag = red + NW * kPanel, *f = flag + kPanel;  // flag[0]: tau of the last step, flag[1]: idle CTAs
    T *V = stage + kStageHead<Team>;
    const int64_t velems = (int64_t)stage_bytes / (int64_t)sizeof(T) - kStageHead<Team>;
    int rank_flag = 0;
    int j0 = j_start;
    while (j0 < p) {
        const int qq = q - j0;
        int nb = (int)min((int64_t)kPanel, velems / (int64_t)max(qq, 1));
        nb = min(nb, p - j0);
        if (nb < 4) {
            householder_step(team, B, q, p, rhs, vhead, taus, j0, j0 + 1, small, rank_flag);
            if (me == 0) {
                pnb[j0] = 1;
                Tst[(int64_t)j0 * kPanel] = taus[j0];
            }
            ++j0;
            continue;
        }
        T *src = B + (int64_t)j0 * q + j0;
        const uint32_t idle = me == 0 ? *(volatile uint32_t *)ho->board.idle : 0u;
        panel_stage(team, src, q, V, qq, nb, (const T *)nullptr);
        if (me == 0) flag[1] = idle ? T(1) : T(0);
        team.sync();
        panel_factor(team, V, qq, nb, src, q, vhead + j0, taus + j0, tm, red, flag, f, small, rank_flag);
        for (int e = me; e < nb * kPanel; e += Team::SIZE) {
            const int t = e / kPanel, s2 = e - t * kPanel;
            Tst[(int64_t)(j0 + t) * kPanel + s2] = (s2 <= t) ? tm[s2 * kPanel + t] : T(0);
        }
        if (me == 0) pnb[j0] = nb;
        wy_apply_shared(team, ho, flag[1] != T(0), V, qq, nb, tm, B, q, p, rhs, j0, j0 + nb, p, vhead + j0,
                        Tst + (int64_t)j0 * kPanel);
        j0 += nb;
    }
    return rank_flag;
}

// The QR update of Section 3, first half: the reflectors 0..p0-1 of a
// finished factor (built on q0 rows; every row below is zero in them) applied
// to the appended columns p0..p-1 of B (ld q), rows j..q0-1, panel by panel as
// they were factored, each panel in compact-WY form with its stored T, split
// into sub-panels when its explicit V outgrows the staging area (q has grown
// since it was factored).  Sub-panels of fewer than four reflectors take one
// reflector at a time, and a run of them goes to update_reflectors together: SPAI's
// factors are nothing but such a run, and a synchronisation per reflector was a tenth of the
// global bin (n = 20000 power law in FP64: 129 -> 120 ms).
template <class Team, typename T>
__device__ __noinline__ void qr_update_apply_staged(Team team, T *B, int q, int p, int q0, int p0, const T *vhead,
                                                    const T *taus, T *stage, int stage_bytes, const T *Tst,
                                                    const int32_t *pnb, HelpOwner *ho) {
    const int me = team.rank();
    T *tm = stage;
    T *flag = stage + kPanel * kPanel + Team::SIZE / 32 * kPanel;
    T *V = stage + kStageHead<Team>;
    const int64_t velems = (int64_t)stage_bytes / (int64_t)sizeof(T) - kStageHead<Team>;
    int j0 = 0, single = 0;  // reflectors single .. j1 - 1 wait for update_reflectors
    while (j0 < p0) {
        const int nb = pnb[j0];
        // the panel in sub-panels of as many reflectors as the staging area holds:
        // the diagonal blocks of a panel's T are the T's of its sub-panels
        for (int js = 0; js < nb;) {
            const int j1 = j0 + js, qq = q0 - j1;
            const int ns = (int)min((int64_t)(nb - js), qq > 0 ? velems / (int64_t)qq : (int64_t)0);
            if (ns < 4) {
                ++js;
                continue;
            }
            if (single < j1) update_reflectors(team, B, q, p, q0, p0, vhead, taus, single, j1);
            single = j1 + ns;
            const T *tcol = Tst + (int64_t)j1 * kPanel + js;
            const uint32_t idle = me == 0 ? *(volatile uint32_t *)ho->board.idle : 0u;
            panel_stage(team, B + (int64_t)j1 * q + j1, (int64_t)q, V, qq, ns, vhead + j1);
            load_T(team, tcol, ns, tm);
            if (me == 0) flag[1] = idle ? T(1) : T(0);
            team.sync();
            wy_apply_shared(team, ho, flag[1] != T(0), V, qq, ns, tm, B, q, p, (T *)nullptr, j1, p0, p - 1,
                            vhead + j1, tcol);
            js += ns;
        }
        j0 += nb;
    }
    if (single < p0) update_reflectors(team, B, q, p, q0, p0, vhead, taus, single, p0);
}

}  // namespace rsai
