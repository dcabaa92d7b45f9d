// bicgstab.cu -- right-preconditioned BiCGStab (Eq. 1.2: A M y = b, x = M y;
// Section 5) as one cooperative kernel: every iteration, its stopping tests and
// the final residual run on the device, and the host waits once.
//
// A solve of a few hundred thousand unknowns is bound by launches and host
// round trips, not by its products (the matrices and vectors stay in L2): as 20
// launches and 3 host reads per iteration, 60 iterations at n = 262144 took
// 13 ms, 220 us each, of which the four products are a quarter.  Here an iteration is seven
// grid-wide barriers.
//
// Where M's rows are long its products take a block per 64 rows and one row per 8 lanes:
// an iteration on power-law matrices 129, 155, 173 -> 77, 99, 119 us (n = 2000, 20000, 60000).
//
// Work split.  Rows go to virtual blocks of 256 rows, dealt out in rounds over
// kDotBlocks of them; a block owns the same rows in every vector step, in A's
// products and in the dot products, so that only M's products (which gather
// from every block) and the sums of the dot products need the whole grid.
//
// Every sum has a fixed order whatever the grid: a product's row on 8 lanes
// and a butterfly; a dot product on kDotBlocks x 256 chains (element b * 256 + t
// + k * kDotBlocks * 256 on chain (b, t), ascending k), a tree per virtual block
// and a tree over the blocks.  Repeated solves give identical iterates.
#include <algorithm>

#include "kernels.h"
#include "spmv.cuh"

namespace rsai {

namespace {

constexpr int kDotBlocks = 304;   // virtual blocks (two per SM)
constexpr int kDotThreads = 256;  // chains per virtual block, and its rows per round
constexpr int kThreads = 512;     // threads per physical block
constexpr int64_t kRound = (int64_t)kDotBlocks * kDotThreads;
// partial sums per iteration: (rhat,r) (rhat,v) (s,s) (t,s) (t,t) (r,r)
enum { D_RHO = 0, D_RV, D_SS, D_TS, D_TT, D_RR, D_COUNT };
// polls of a barrier before it is given up (about a microsecond each)
constexpr unsigned kBarrierPolls = 1u << 24;

struct Control {          // zeroed before the launch
    unsigned arrived;     // barrier arrivals so far
    unsigned timeout;     // a barrier was given up
    int status, iters;
    double relres;
};
constexpr int kControlWords = 8;
static_assert(sizeof(Control) <= kControlWords * sizeof(double), "control block");

struct Solve {
    int64_t n;
    int vblocks;  // virtual blocks that hold rows
    CsrView A, M;
    bool long_A, long_M;  // rows of kLongAverage entries and more on the average
    const double *b;
    double *x;
    double *r, *rhat, *p, *v, *s, *t, *y, *tmp, *tmp2, *partials;
    Control *ctl;
    double rtol;
    int maxit;
};

// Grid-wide barrier (cooperative launch: every block is resident).  Bounded:
// returns false once any block has given up, and the caller returns.
__device__ bool grid_sync(Control *ctl, unsigned &epoch) {
    __shared__ int ok_sh;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        const unsigned goal = ++epoch * gridDim.x;
        atomicAdd(&ctl->arrived, 1u);
        int ok = 1;
        unsigned seen = 0, polls = 0;
        for (;;) {
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(seen) : "l"(&ctl->arrived) : "memory");
            if ((int)(seen - goal) >= 0) break;
            if (++polls >= kBarrierPolls || *(volatile unsigned *)&ctl->timeout != 0u) {
                atomicExch(&ctl->timeout, 1u);
                ok = 0;
                break;
            }
        }
        __threadfence();
        ok_sh = ok;
    }
    __syncthreads();
    return ok_sh != 0;
}

// y[r0 .. end) = (A x) of these rows by one block, four rows per 8 lanes, or one where rows are long
constexpr int kGroups = kThreads / 8;
static_assert(kGroups * 4 == kDotThreads, "one round of a virtual block is one pass of a block");
__device__ __forceinline__ void block_rows(const CsrView &A, bool is_long, const double *x, double *y, int64_t r0,
                                           int64_t end) {
    const int g = threadIdx.x >> 3, sub = threadIdx.x & 7;
    if (is_long) {
        for (; r0 < end; r0 += kGroups) spmv_row<2>(A, x, y, r0 + g, r0 + g < end, sub);
    } else {
        // without the next round's loads ahead, which k_spmv gains from: here they cost the rest
        // of the kernel registers (2-D stencil with 80089 unknowns 77.7 -> 79.2 us per iteration)
        for (; r0 < end; r0 += kGroups * 4)
            spmv_long_rows<4>(A, x, y, r0 + g * 4, spmv_short_rows<4, false>(A, x, y, r0 + g * 4, end, sub), sub);
    }
}

// y = A x, an even share of the rows per block
__device__ void product(const CsrView &A, bool is_long, int64_t n, const double *x, double *y) {
    const int64_t share = ((n + gridDim.x - 1) / gridDim.x + 3) / 4 * 4;
    block_rows(A, is_long, x, y, blockIdx.x * share, min(n, (blockIdx.x + 1) * share));
}

// y = A x on the rows that this block owns
__device__ void product_own(const Solve &S, const double *x, double *y) {
    for (int vb = blockIdx.x; vb < S.vblocks; vb += gridDim.x)
        for (int64_t r0 = (int64_t)vb * kDotThreads; r0 < S.n; r0 += kRound)
            block_rows(S.A, S.long_A, x, y, r0, min(S.n, r0 + kDotThreads));
    __syncthreads();
}

// Operands of up to two dot products of four rounds of a virtual block
struct Shared {
    double x[2][4][kDotThreads], y[2][4][kDotThreads];
    double tree[2][kDotThreads];
    double scalar;
};

// f(i, x, y) over the elements that this block owns (all threads; x and y get
// the operands of ND dot products), and the partial sums of the products: four
// rounds at a time are formed by all threads, then each chain adds its four
// products in order; the tree over the 256 chains of a virtual block last.
template <int ND, typename F> __device__ void chains(const Solve &S, Shared &sh, const int (&d)[ND], F f) {
    const int t = threadIdx.x % kDotThreads, g = threadIdx.x / kDotThreads;
    for (int vb = blockIdx.x; vb < S.vblocks; vb += gridDim.x) {
        double acc[ND];
#pragma unroll
        for (int q = 0; q < ND; ++q) acc[q] = 0.0;
        for (int64_t r0 = (int64_t)vb * kDotThreads; r0 < S.n; r0 += 4 * kRound) {
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int k = g + 2 * h;
                const int64_t i = r0 + k * kRound + t;
                double x[ND], y[ND];
#pragma unroll
                for (int q = 0; q < ND; ++q) x[q] = y[q] = 0.0;
                if (i < S.n) f(i, x, y);
#pragma unroll
                for (int q = 0; q < ND; ++q) {
                    sh.x[q][k][t] = x[q];
                    sh.y[q][k][t] = y[q];
                }
            }
            __syncthreads();
            // dot product q on threads q * 256 ...
            if (g < ND) {
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    if (r0 + k * kRound + t < S.n) {
#pragma unroll
                        for (int q = 0; q < ND; ++q)
                            if (g == q) acc[0] = fma(sh.x[q][k][t], sh.y[q][k][t], acc[0]);
                    }
                }
            }
            __syncthreads();
        }
        if (g < ND) sh.tree[g][t] = acc[0];
        __syncthreads();
        for (int o = kDotThreads / 2; o > 0; o >>= 1) {
            if (g < ND && t < o) sh.tree[g][t] += sh.tree[g][t + o];
            __syncthreads();
        }
        if (g < ND && t == 0) S.partials[(int64_t)d[g < ND ? g : 0] * kDotBlocks + vb] = sh.tree[g][0];
        __syncthreads();
    }
}

// The sum of a dot product's partials, by every block (a tree over 512 slots of
// which kDotBlocks hold a partial sum); the result to every thread
__device__ double grid_total(const double *partials, Shared &sh) {
    double *s = sh.tree[0];
    const int t = threadIdx.x;
    if (t < 256) {
        double v = t < kDotBlocks ? partials[t] : 0.0;
        v += t + 256 < kDotBlocks ? partials[t + 256] : 0.0;
        s[t] = v;
    }
    __syncthreads();
    for (int o = 128; o > 0; o >>= 1) {
        if (t < o) s[t] += s[t + o];
        __syncthreads();
    }
    const double v = s[0];
    __syncthreads();
    return v;
}

// f() by one thread, its value to all.  An FP64 division or square root by
// every thread of the grid would take the FP64 units longer than a product with A.
template <typename F> __device__ __forceinline__ double block_scalar(Shared &sh, F f) {
    if (threadIdx.x == 0) sh.scalar = f();
    __syncthreads();
    const double v = sh.scalar;
    __syncthreads();
    return v;
}

// f(i) over the elements that this block owns, all threads
template <typename F> __device__ void own_elements(const Solve &S, F f) {
    constexpr int G = kThreads / kDotThreads;
    for (int vb = blockIdx.x; vb < S.vblocks; vb += gridDim.x)
        for (int64_t r0 = (int64_t)vb * kDotThreads + (threadIdx.x / kDotThreads) * kRound; r0 < S.n; r0 += G * kRound) {
            const int64_t i = r0 + threadIdx.x % kDotThreads;
            if (i < S.n) f(i);
        }
}

__global__ void __launch_bounds__(kThreads, 2) k_bicgstab(Solve S) {
    __shared__ Shared sh;
    const int64_t n = S.n;
    Control *ctl = S.ctl;
    unsigned epoch = 0;
    const bool prec = S.M.row_ptr != nullptr;
    const double *P = S.partials;
#define RSAI_SYNC() \
    do { if (!grid_sync(ctl, epoch)) return; } while (0)
    own_elements(S, [&](int64_t i) {
        const double bi = S.b[i];
        S.r[i] = bi;
        S.rhat[i] = bi;
        S.p[i] = 0.0;
        S.v[i] = 0.0;
        S.y[i] = 0.0;
    });
    __syncthreads();
    chains<1>(S, sh, {D_RHO}, [&](int64_t i, double (&a)[1], double (&c)[1]) {
        a[0] = S.rhat[i];
        c[0] = S.r[i];
    });
    RSAI_SYNC();
    // r = rhat = b: (rhat,r) is also (b,b)
    double rho = grid_total(P + D_RHO * kDotBlocks, sh);
    const double nb = block_scalar(sh, [&] { return sqrt(rho); });
    if (nb == 0.0) {
        own_elements(S, [&](int64_t i) { S.x[i] = 0.0; });
        if (blockIdx.x == 0 && threadIdx.x == 0) {
            ctl->status = RSAI_OK;
            ctl->iters = 0;
            ctl->relres = 0.0;
        }
        return;
    }
    double rho_old = 1.0, alpha = 1.0, omega = 1.0;
    int status = RSAI_ERR_NOT_CONVERGED, it = 1;
    for (; it <= S.maxit; ++it) {
        const double beta = block_scalar(sh, [&] { return (rho / rho_old) * (alpha / omega); });
        own_elements(S, [&](int64_t i) {
            S.p[i] = S.r[i] + beta * (S.p[i] - omega * S.v[i]);
        });
        const double *Mp = S.p;
        RSAI_SYNC();
        if (prec) {
            product(S.M, S.long_M, n, S.p, S.tmp);
            Mp = S.tmp;
            RSAI_SYNC();
        }
        product_own(S, Mp, S.v);
        chains<1>(S, sh, {D_RV}, [&](int64_t i, double (&a)[1], double (&c)[1]) {
            a[0] = S.rhat[i];
            c[0] = S.v[i];
        });
        RSAI_SYNC();
        const double rv = grid_total(P + D_RV * kDotBlocks, sh);
        alpha = block_scalar(sh, [&] { return rho / rv; });
        chains<1>(S, sh, {D_SS}, [&](int64_t i, double (&a)[1], double (&c)[1]) {
            const double si = S.r[i] - alpha * S.v[i];
            S.s[i] = si;
            a[0] = c[0] = si;
        });
        RSAI_SYNC();
        const double ss = grid_total(P + D_SS * kDotBlocks, sh);
        // rho = r^T r = 0, or r^T v = 0 (alpha undefined): the recurrences break down
        if (rho == 0.0 || rv == 0.0) { status = RSAI_ERR_BREAKDOWN; break; }
        if (block_scalar(sh, [&] { return sqrt(ss) / nb; }) < S.rtol) {
            own_elements(S, [&](int64_t i) { S.y[i] += alpha * S.p[i]; });
            status = RSAI_OK;
            break;
        }
        const double *Ms = S.s;
        if (prec) {
            product(S.M, S.long_M, n, S.s, S.tmp);
            Ms = S.tmp;
            RSAI_SYNC();
        }
        product_own(S, Ms, S.t);
        chains<2>(S, sh, {D_TS, D_TT}, [&](int64_t i, double (&a)[2], double (&c)[2]) {
            a[0] = a[1] = c[1] = S.t[i];
            c[0] = S.s[i];
        });
        RSAI_SYNC();
        const double ts = grid_total(P + D_TS * kDotBlocks, sh), tt = grid_total(P + D_TT * kDotBlocks, sh);
        if (tt == 0.0) { status = RSAI_ERR_BREAKDOWN; break; }
        omega = block_scalar(sh, [&] { return ts / tt; });
        chains<2>(S, sh, {D_RR, D_RHO}, [&](int64_t i, double (&a)[2], double (&c)[2]) {
            S.y[i] += alpha * S.p[i] + omega * S.s[i];
            const double ri = S.s[i] - omega * S.t[i];
            S.r[i] = ri;
            a[0] = c[0] = c[1] = ri;
            a[1] = S.rhat[i];
        });
        RSAI_SYNC();
        const double rr = grid_total(P + D_RR * kDotBlocks, sh);
        if (block_scalar(sh, [&] { return sqrt(rr) / nb; }) < S.rtol) { status = RSAI_OK; break; }
        if (omega == 0.0) { status = RSAI_ERR_BREAKDOWN; break; }
        rho_old = rho;
        rho = grid_total(P + D_RHO * kDotBlocks, sh);
    }
    if (it > S.maxit) it = S.maxit;
    // x = M y, true residual
    RSAI_SYNC();
    if (prec) product(S.M, S.long_M, n, S.y, S.x);
    else own_elements(S, [&](int64_t i) { S.x[i] = S.y[i]; });
    RSAI_SYNC();
    product_own(S, S.x, S.tmp2);
    chains<1>(S, sh, {D_RV}, [&](int64_t i, double (&a)[1], double (&c)[1]) { a[0] = c[0] = S.b[i] - S.tmp2[i]; });
    RSAI_SYNC();
    const double res = grid_total(P + D_RV * kDotBlocks, sh);
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        ctl->status = status;
        ctl->iters = it;
        ctl->relres = sqrt(res) / nb;
    }
#undef RSAI_SYNC
}

}  // namespace

size_t bicgstab_workspace_bytes(int64_t n) {
    return sizeof(double) * ((size_t)(n > 0 ? n : 1) * 9 + (size_t)D_COUNT * kDotBlocks + kControlWords);
}

int bicgstab_run(int64_t n, int64_t nnzA, const int64_t *Arp, const int32_t *Aci, const double *Av, int64_t nnzM,
                 const int64_t *Mrp, const int32_t *Mci, const double *Mv, const double *b, double *x, double rtol, int maxit,
                 int *iters, double *relres, cudaStream_t st, double *work) {
    double *buf = work;
    const bool own = work == nullptr;  // else the caller's workspace of bicgstab_workspace_bytes(n)
    if (own && cudaMallocAsync((void **)&buf, bicgstab_workspace_bytes(n), st) != cudaSuccess)
        return RSAI_ERR_OOM;
    Solve S{};
    S.n = n;
    S.vblocks = (int)std::min<int64_t>(kDotBlocks, (n + kDotThreads - 1) / kDotThreads);
    S.A = CsrView{Arp, Aci, Av};
    S.M = CsrView{Mrp, Mci, Mv};
    S.long_A = nnzA / n >= kLongAverage;
    S.long_M = Mrp && nnzM / n >= kLongAverage;
    S.b = b;
    S.x = x;
    double *q = buf;
    for (double **v : {&S.r, &S.rhat, &S.p, &S.v, &S.s, &S.t, &S.y, &S.tmp, &S.tmp2}) {
        *v = q;
        q += n;
    }
    S.partials = q;
    S.ctl = reinterpret_cast<Control *>(q + (size_t)D_COUNT * kDotBlocks);
    S.rtol = rtol;
    S.maxit = maxit;
    int dev = 0, sms = 0, occ = 0;
    Control c{};
    auto run = [&]() -> bool {
        if (cudaGetDevice(&dev) != cudaSuccess ||
            cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_bicgstab, kThreads, 0) != cudaSuccess || occ < 1)
            return false;
        // a block per virtual block or, where M's rows are long, one per 64 rows of it (a pass of its
        // groups): blocks beyond the virtual ones take part in M's products only
        const int64_t want = std::max<int64_t>(S.vblocks, S.long_M ? (n + kGroups - 1) / kGroups : 1);
        const int grid = (int)std::max<int64_t>(1, std::min<int64_t>({want, kDotBlocks, (int64_t)occ * sms}));
        // partial sums of virtual blocks without rows, and the control block
        if (cudaMemsetAsync(S.partials, 0, sizeof(double) * ((size_t)D_COUNT * kDotBlocks + kControlWords), st) !=
            cudaSuccess)
            return false;
        void *args[] = {&S};
        if (cudaLaunchCooperativeKernel((const void *)k_bicgstab, dim3(grid), dim3(kThreads), args, 0, st) !=
            cudaSuccess)
            return false;
        return cudaMemcpyAsync(&c, S.ctl, sizeof(c), cudaMemcpyDeviceToHost, st) == cudaSuccess;
    };
    const bool ok = run();
    if (!ok) cudaGetLastError();
    if (own) cudaFreeAsync(buf, st);
    if (!ok || cudaStreamSynchronize(st) != cudaSuccess) return RSAI_ERR_CUDA;
    if (c.timeout) return RSAI_ERR_TIMEOUT;
    *iters = c.iters;
    *relres = c.relres;
    return c.status;
}

}  // namespace rsai
