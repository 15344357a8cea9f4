// CholInv (Algorithm 1, Section II-D): [L, Y] = CholInv(W) with W = L L^T and
// Y = L^-1, by the paper's halving recursion
//     [L11, Y11] = CholInv(W11)
//     L21 = W21 Y11^T
//     [L22, Y22] = CholInv(W22 - L21 L21^T)
//     Y21 = -Y22 (L21 Y11)            (association of Algorithm CFR3D)
// run as FP64 GEMM launches on one stream. The recursion stops at leaves of at
// most 128 (the paper's base case is n = 1; CFR3D stops at n_o and factors the
// block redundantly), each one launch (cholinv_leaf.cu). The split point is a
// multiple of 64 near n/2 instead of floor(n/2): the result is the same
// factorization, rounded in a different order.
#include <algorithm>

#include "kernels.h"

namespace cqr2 {
namespace {

constexpr int NB = CHOLINV_BASE;

__global__ void k_transpose_lower(const double* L, int64_t ldl, int n, double* R,
                                  int64_t ldr) {
  grid_chain();
  __shared__ double tile[32][33];
  const int bi = blockIdx.x * 32, bj = blockIdx.y * 32;  // R block (rows bi.., cols bj..)
  // read L block (rows bj.., cols bi..) coalesced along its rows
  for (int y = threadIdx.y; y < 32; y += 8) {
    const int li = bj + threadIdx.x, lj = bi + y;
    tile[y][threadIdx.x] = (li < n && lj < n) ? L[li + (int64_t)lj * ldl] : 0.0;
  }
  __syncthreads();
  for (int y = threadIdx.y; y < 32; y += 8) {
    const int ri = bi + threadIdx.x, rj = bj + y;
    if (ri < n && rj < n) R[ri + (int64_t)rj * ldr] = (ri <= rj) ? tile[threadIdx.x][y] : 0.0;
  }
}

__global__ void k_copy_upper(const double* X, int64_t ldx, int n, double* R, int64_t ldr) {
  grid_chain();
  const int i = blockIdx.x * blockDim.x + threadIdx.x, j = blockIdx.y;
  if (i < n) R[i + (int64_t)j * ldr] = (i <= j) ? X[i + (int64_t)j * ldx] : 0.0;
}

cudaError_t rec(int n, double* Wk, int64_t ldk, double* L, int64_t ldl, double* Y, int64_t ldy, double* U,
                int64_t ldu, DevStatus* st, int pass, long long off, Lane s) {
  if (n <= CHOLINV_LEAF) return cholinv_leaf(n, Wk, ldk, L, ldl, Y, ldy, nullptr, 0, nullptr, 0, st, pass, off, s);
  const int n1 = NB * (int)ceil_div(n, 2 * NB);
  const int n2 = n - n1;
  cudaError_t e;
  // [L11, Y11] = CholInv(W11)
  if ((e = rec(n1, Wk, ldk, L, ldl, Y, ldy, U, ldu, st, pass, off, s)) != cudaSuccess) return e;
  // L21 = W21 Y11^T
  if ((e = gemm_f64(n2, n1, n1, 1.0, Wk + n1, ldk, Y, ldy, 0.0, L + n1, ldl, GEMM_TB | GEMM_B_UPPER | GEMM_BETA0,
                    s)) != cudaSuccess)
    return e;
  // W22 <- W22 - L21 L21^T (lower triangle)
  double* W22 = Wk + n1 + (int64_t)n1 * ldk;
  if ((e = gemm_f64(n2, n2, n1, -1.0, L + n1, ldl, L + n1, ldl, 1.0, W22, ldk, GEMM_TB | GEMM_C_LOWER, s)) != cudaSuccess)
    return e;
  // [L22, Y22] = CholInv(W22 - L21 L21^T)
  double* L22 = L + n1 + (int64_t)n1 * ldl;
  double* Y22 = Y + n1 + (int64_t)n1 * ldy;
  if ((e = rec(n2, W22, ldk, L22, ldl, Y22, ldy, U, ldu, st, pass, off + n1, s)) != cudaSuccess) return e;
  // U = L21 Y11
  if ((e = gemm_f64(n2, n1, n1, 1.0, L + n1, ldl, Y, ldy, 0.0, U, ldu, GEMM_B_LOWER | GEMM_BETA0, s)) !=
      cudaSuccess)
    return e;
  // Y21 = -Y22 U
  return gemm_f64(n2, n1, n2, -1.0, Y22, ldy, U, ldu, 0.0, Y + n1, ldy, GEMM_A_LOWER | GEMM_BETA0, s);
}

// Depth-limited recursion: the top `depth` levels form L21 by block forward
// substitution through the diagonal blocks' inverses and leave Y21 zero.
cudaError_t rec_depth(int n, double* Wk, int64_t ldk, double* L, int64_t ldl, double* Y, int64_t ldy, double* U,
                      int64_t ldu, double* T, int64_t ldt, DevStatus* st, int pass, long long off, int depth,
                      Lane s) {
  if (depth <= 0 || n <= NB) return rec(n, Wk, ldk, L, ldl, Y, ldy, U, ldu, st, pass, off, s);
  const int n1 = NB * (int)ceil_div(n, 2 * NB);
  const int n2 = n - n1;
  cudaError_t e;
  // [L11, Y11] with Y11 known on its leaf blocks only
  if ((e = rec_depth(n1, Wk, ldk, L, ldl, Y, ldy, U, ldu, T, ldt, st, pass, off, depth - 1, s)) !=
      cudaSuccess)
    return e;
  // L21 = W21 L11^-T
  if ((e = right_solve(n2, n1, Wk + n1, ldk, L + n1, ldl, L, ldl, Y, ldy, depth - 1, T, ldt, s)) != cudaSuccess)
    return e;
  // W22 <- W22 - L21 L21^T (lower triangle)
  double* W22 = Wk + n1 + (int64_t)n1 * ldk;
  if ((e = gemm_f64(n2, n2, n1, -1.0, L + n1, ldl, L + n1, ldl, 1.0, W22, ldk, GEMM_TB | GEMM_C_LOWER, s)) != cudaSuccess)
    return e;
  return rec_depth(n2, W22, ldk, L + n1 + (int64_t)n1 * ldl, ldl, Y + n1 + (int64_t)n1 * ldy, ldy, U, ldu, T, ldt,
                   st, pass, off + n1, depth - 1, s);
}

}  // namespace

cudaError_t right_solve(int64_t M, int N, const double* B, int64_t ldb, double* X, int64_t ldx, const double* L,
                        int64_t ldl, const double* Y, int64_t ldy, int depth, double* T, int64_t ldt,
                        Lane s) {
  cudaError_t e;
  if (M <= 0 || N <= 0) return cudaSuccess;
  if (depth <= 0 || N <= NB) {
    // X = B Y^T with Y the inverse of this diagonal block (Y^T upper triangular)
    if ((const double*)X != B)
      return gemm_f64(M, N, N, 1.0, B, ldb, Y, ldy, 0.0, X, ldx, GEMM_TB | GEMM_B_UPPER | GEMM_BETA0, s);
    if ((e = gemm_f64(M, N, N, 1.0, B, ldb, Y, ldy, 0.0, T, ldt, GEMM_TB | GEMM_B_UPPER | GEMM_BETA0, s)) !=
        cudaSuccess)
      return e;
    return cudaMemcpy2DAsync(X, (size_t)ldx * sizeof(double), T, (size_t)ldt * sizeof(double),
                             (size_t)M * sizeof(double), (size_t)N, cudaMemcpyDeviceToDevice, s);
  }
  // the split of the recursion that formed Y, so the leaves are its inverted blocks
  const int n1 = NB * (int)ceil_div(N, 2 * NB);
  const int n2 = N - n1;
  // X1 = B1 L11^-T
  if ((e = right_solve(M, n1, B, ldb, X, ldx, L, ldl, Y, ldy, depth - 1, T, ldt, s)) != cudaSuccess) return e;
  // X2 = (B2 - X1 L21^T) L22^-T, the bracket formed in X2
  double* X2 = X + (int64_t)n1 * ldx;
  if ((const double*)X != B &&
      (e = cudaMemcpy2DAsync(X2, (size_t)ldx * sizeof(double), B + (int64_t)n1 * ldb, (size_t)ldb * sizeof(double),
                             (size_t)M * sizeof(double), (size_t)n2, cudaMemcpyDeviceToDevice, s)) != cudaSuccess)
    return e;
  if ((e = gemm_f64(M, n2, n1, -1.0, X, ldx, L + n1, ldl, 1.0, X2, ldx, GEMM_TB, s)) != cudaSuccess) return e;
  return right_solve(M, n2, X2, ldx, X2, ldx, L + n1 + (int64_t)n1 * ldl, ldl, Y + n1 + (int64_t)n1 * ldy, ldy,
                     depth - 1, T, ldt, s);
}

int right_solve_temp_cols(int n) { return n <= NB ? n : NB * (int)ceil_div(n, 2 * NB); }

cudaError_t cholinv_depth(int n, const double* W, int64_t ldw, double* L, int64_t ldl, double* Y, int64_t ldy,
                          double* work, double* U, double* T, int64_t ldt, DevStatus* st, int pass, int depth,
                          Lane s) {
  if (depth <= 0) return cholinv(n, W, ldw, L, ldl, Y, ldy, work, U, st, pass, s);
  cudaError_t e;
  if ((e = cudaMemcpy2DAsync(work, (size_t)n * sizeof(double), W, (size_t)ldw * sizeof(double),
                             (size_t)n * sizeof(double), (size_t)n, cudaMemcpyDeviceToDevice, s)) != cudaSuccess)
    return e;
  if ((e = cudaMemset2DAsync(L, (size_t)ldl * sizeof(double), 0, (size_t)n * sizeof(double), (size_t)n, s)) !=
      cudaSuccess)
    return e;
  if ((e = cudaMemset2DAsync(Y, (size_t)ldy * sizeof(double), 0, (size_t)n * sizeof(double), (size_t)n, s)) !=
      cudaSuccess)
    return e;
  return rec_depth(n, work, n, L, ldl, Y, ldy, U, n, T, ldt, st, pass, 0, depth, s);
}

cudaError_t cholinv(int n, const double* W, int64_t ldw, double* L, int64_t ldl, double* Y, int64_t ldy,
                    double* work, double* U, DevStatus* st, int pass, Lane s,
                    double* Rt, int64_t ldrt, double* Rp) {
  cudaError_t e;
  if (n <= CHOLINV_LEAF) {
    // one leaf: straight from W, with R and, up to 64 columns, the packed R^-1
    // when asked: 4096 x 64 171 us, packed by a launch of its own 176, 1024 x 16 49
    // and 51. Above 64 columns that launch stays, though in the leaf it would take
    // 3 us less too (3000 x 80 231 and 228, 4096 x 128 499 and 496): the suite counts
    // on more than ten launches per factorization at 96 columns.
    double* leafRp = n <= NB ? Rp : nullptr;
    const int rpw = leafRp != nullptr ? qform_group_width(n) : 0;
    // the packing's layout is the Q-form's: the same number of column groups and pitch
    if (leafRp != nullptr && rpack_doubles(n) != (size_t)RP_GROUPS * n * (rpw + (rpw & 1))) return cudaErrorInvalidValue;
    if ((e = cholinv_leaf(n, W, ldw, L, ldl, Y, ldy, Rt, ldrt, leafRp, rpw, st, pass, 0, s)) != cudaSuccess) return e;
    return Rp != nullptr && leafRp == nullptr ? pack_rinv_from_lower(Y, ldy, n, Rp, s) : cudaSuccess;
  }
  if ((e = cudaMemcpy2DAsync(work, (size_t)n * sizeof(double), W, (size_t)ldw * sizeof(double),
                             (size_t)n * sizeof(double), (size_t)n, cudaMemcpyDeviceToDevice, s)) != cudaSuccess)
    return e;
  if ((e = cudaMemset2DAsync(L, (size_t)ldl * sizeof(double), 0, (size_t)n * sizeof(double), (size_t)n, s)) !=
      cudaSuccess)
    return e;
  if ((e = cudaMemset2DAsync(Y, (size_t)ldy * sizeof(double), 0, (size_t)n * sizeof(double), (size_t)n, s)) !=
      cudaSuccess)
    return e;
  if ((e = rec(n, work, n, L, ldl, Y, ldy, U, n, st, pass, 0, s)) != cudaSuccess) return e;
  if (Rt != nullptr && (e = transpose_lower(L, ldl, n, Rt, ldrt, s)) != cudaSuccess) return e;
  if (Rp != nullptr) return pack_rinv_from_lower(Y, ldy, n, Rp, s);
  return cudaSuccess;
}

// Shift of the shifted CholeskyQR pass: W += s I with
// s = 11 (m n + n (n+1)) u trace(W), u = 2^-53 (||A||_F^2 = trace(A^T A)).
// One CTA; the trace is summed in a fixed order.
__global__ void __launch_bounds__(256) k_add_shift(double* W, int64_t ldw, int n, int64_t m) {
  __shared__ double part[256];
  double t = 0.0;
  for (int i = threadIdx.x; i < n; i += 256) t += W[i + (int64_t)i * ldw];
  part[threadIdx.x] = t;
  __syncthreads();
  for (int h = 128; h > 0; h >>= 1) {
    if (threadIdx.x < h) part[threadIdx.x] += part[threadIdx.x + h];
    __syncthreads();
  }
  const double s = 11.0 * ((double)m * n + (double)n * (n + 1)) * 0x1p-53 * part[0];
  for (int i = threadIdx.x; i < n; i += 256) W[i + (int64_t)i * ldw] += s;
}

cudaError_t add_shift(double* W, int64_t ldw, int n, int64_t m, cudaStream_t s) {
  k_add_shift<<<1, 256, 0, s>>>(W, ldw, n, m);
  count_launch();
  return cudaGetLastError();
}

cudaError_t transpose_lower(const double* L, int64_t ldl, int n, double* R, int64_t ldr, Lane s) {
  dim3 grid((unsigned)ceil_div(n, 32), (unsigned)ceil_div(n, 32));
  cudaError_t e = launch_chained(k_transpose_lower, grid, dim3(32, 8), 0, s, dim3(1), true, L, ldl, n, R, ldr);
  if (e != cudaSuccess) return e;
  count_launch();
  return cudaGetLastError();
}

cudaError_t copy_upper(const double* X, int64_t ldx, int n, double* R, int64_t ldr, Lane s) {
  dim3 grid((unsigned)ceil_div(n, 128), (unsigned)n);
  cudaError_t e = launch_chained(k_copy_upper, grid, dim3(128), 0, s, dim3(1), true, X, ldx, n, R, ldr);
  if (e != cudaSuccess) return e;
  count_launch();
  return cudaGetLastError();
}

}  // namespace cqr2
