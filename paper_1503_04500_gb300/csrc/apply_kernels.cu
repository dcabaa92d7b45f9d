// apply_kernels.cu -- CSR SpMV (y = M x, y = A x) and its adjoint in the values
// (the preconditioned solve is in bicgstab.cu).
#include "kernels.h"
#include "spmv.cuh"

namespace rsai {

// R rows per 8 lanes; 128 threads per CTA spread the groups with long rows better than 256
constexpr int kSpmvThreads = 128;
template <int R>
__global__ void __launch_bounds__(kSpmvThreads)
    k_spmv(int64_t n, CsrView A, const double *__restrict__ x, double *__restrict__ y) {
    const int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int sub = threadIdx.x & 7;
    const int64_t row0 = (g >> 3) * R;
    if constexpr (R == 1) spmv_row<2>(A, x, y, row0, row0 < n, sub);
    else spmv_long_rows<R>(A, x, y, row0, spmv_short_rows<R>(A, x, y, row0, n, sub), sub);
}

// gval[e] = gy[i] x[col(e)] for every stored entry e of row i: the gradient
// of y = A x with respect to the stored values of A.  8 lanes per row, one
// write per entry, no reduction.
__global__ void k_spmv_grad_values(int64_t n, const int64_t *__restrict__ row_ptr,
                                   const int32_t *__restrict__ col_idx, const double *__restrict__ gy,
                                   const double *__restrict__ x, double *__restrict__ gval) {
    int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    int64_t row = g >> 3;
    int sub = threadIdx.x & 7;
    if (row >= n) return;
    const double gr = gy[row];
    const int64_t a = row_ptr[row], b = row_ptr[row + 1];
    for (int64_t e = a + sub; e < b; e += 8) gval[e] = gr * x[col_idx[e]];
}

cudaError_t launch_spmv_grad_values(int64_t n, const int64_t *row_ptr, const int32_t *col_idx, const double *gy,
                                    const double *x, double *gval, cudaStream_t st) {
    if (n == 0) return cudaSuccess;
    const int T = 256;
    k_spmv_grad_values<<<(unsigned)((n * 8 + T - 1) / T), T, 0, st>>>(n, row_ptr, col_idx, gy, x, gval);
    return cudaGetLastError();
}

cudaError_t launch_spmv(int64_t n, int64_t nnz, const int64_t *row_ptr, const int32_t *col_idx, const double *val,
                        const double *x, double *y, cudaStream_t st) {
    if (n == 0) return cudaSuccess;
    const int R = spmv_rows_per_group(n, nnz);
    const int64_t groups = (n + R - 1) / R;
    const unsigned grid = (unsigned)((groups * 8 + kSpmvThreads - 1) / kSpmvThreads);
    const CsrView A{row_ptr, col_idx, val};
    if (R == 1) k_spmv<1><<<grid, kSpmvThreads, 0, st>>>(n, A, x, y);
    else if (R == 2) k_spmv<2><<<grid, kSpmvThreads, 0, st>>>(n, A, x, y);
    else k_spmv<4><<<grid, kSpmvThreads, 0, st>>>(n, A, x, y);
    return cudaGetLastError();
}

}  // namespace rsai
