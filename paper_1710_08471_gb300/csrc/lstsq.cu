// Least-squares tail x = R^-1 (Q^T b). The paper uses QR for least squares
// (Section I) but gives no solve; this library forms c = Q^T b with split-m
// partial sums (summed in a fixed order) and solves R x = c by back
// substitution in one CTA.
#include <algorithm>
#include <type_traits>

#include "fp64_rsqrt.cuh"
#include "kernels.h"

namespace cqr2 {
namespace {

// c = Q^T b as partial sums over row ranges. One FMA per entry of Q makes the
// FP64 pipe the bound (one warp instruction per 16 clocks per SM: 57 us for
// 131601 x 256, where the 270 MB of Q take 40 us), so everything else has to
// stay off it and the loads have to be deep enough to feed it:
//  - a warp owns GC = 8 columns and one row range, so b is loaded once for
//    eight FMAs and 16 loads of Q are in flight per lane (unroll 2);
//  - the eight 32-lane sums are reduced together, each exchange halving the
//    number of live vectors (4 + 2 + 1 + 1 + 1 additions for eight columns,
//    where a butterfly per column takes 40);
//  - a CTA's eight warps take up to eight column groups, and where there are
//    fewer (n <= 32) the rest of the warps take more row ranges.
// 131601 x 256: 280 -> 69 us (83% of the FP64 pipe); 50021 x 100: 86 -> 15 us.
constexpr int GT = 256, GW = GT / 32, GC = 8;

__global__ void __launch_bounds__(GT) k_gemv_t_partial(const double* Q, int64_t ldq, int64_t m, int n,
                                                       const double* b, int64_t rows_per, int gpc,
                                                       double* partial) {
  grid_chain();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t split = (int64_t)blockIdx.x * (GW / gpc) + warp / gpc;
  const int c0 = ((int)blockIdx.y * gpc + warp % gpc) * GC;
  if (c0 >= n) return;
  const int64_t r0 = split * rows_per;
  const int64_t r1 = min(m, r0 + rows_per);
  const double* q[GC];  // columns past n repeat the last one (not stored)
#pragma unroll
  for (int c = 0; c < GC; ++c) q[c] = Q + (int64_t)min(c0 + c, n - 1) * ldq;
  double s[GC];
#pragma unroll
  for (int c = 0; c < GC; ++c) s[c] = 0.0;
  int64_t r = r0 + lane;
  for (; r + 32 < r1; r += 64) {
    double v[2][GC];
    const double b0 = b[r], b1 = b[r + 32];
#pragma unroll
    for (int c = 0; c < GC; ++c) {
      v[0][c] = q[c][r];
      v[1][c] = q[c][r + 32];
    }
#pragma unroll
    for (int c = 0; c < GC; ++c) s[c] = fma(v[0][c], b0, s[c]);
#pragma unroll
    for (int c = 0; c < GC; ++c) s[c] = fma(v[1][c], b1, s[c]);
  }
  if (r < r1) {
    const double b0 = b[r];
#pragma unroll
    for (int c = 0; c < GC; ++c) s[c] = fma(q[c][r], b0, s[c]);
  }
  __syncwarp();
  // lanes with bit h set keep the upper half of the live columns
#pragma unroll
  for (int h = GC / 2, bit = 16; h >= 1; h >>= 1, bit >>= 1) {
    const bool up = (lane & bit) != 0;
#pragma unroll
    for (int c = 0; c < h; ++c) {
      const double keep = up ? s[c + h] : s[c], send = up ? s[c] : s[c + h];
      s[c] = keep + __shfl_xor_sync(0xffffffffu, send, bit);
    }
  }
  s[0] += __shfl_xor_sync(0xffffffffu, s[0], 2);
  s[0] += __shfl_xor_sync(0xffffffffu, s[0], 1);
  const int col = c0 + (lane >> 2);  // lane bits 16, 8, 4 chose the column's bits 4, 2, 1
  if ((lane & 3) == 0 && col < n) partial[split * n + col] = s[0];
}

// x solves R x = c, one CTA, blocked by 32 columns from the right. A column
// at a time cost a division (some 700 clocks of dependent FP64 operations)
// and two block barriers per column; here
//  - the partial sums of c are added by all threads (a fixed split, then a
//    fixed order);
//  - one warp solves the 32 x 32 diagonal block from registers, in the form
//    c_i -= (R_ik / R_kk) c_k, so that a column's chain is a shuffle and an
//    FMA, and x = c / R_kk comes last, for all columns at once. The quotients
//    are correctly rounded, from the diagonal's reciprocals and a correction
//    each (products with the reciprocals alone: 0.8 us less at 16 columns and
//    2 us at 32, none at 100 and more, and at 16 columns an error of the solve
//    9% above that with divisions). Two warps take
//    the blocks in turn: one loads and scales its next block while the other
//    solves (where an entry is too small or too large for this, the block is
//    solved with divisions);
//  - the other warps then update the rows above the block, two lanes to a row
//    with 16 values of R each, loaded ahead of the barrier.
// Now 60 us at n = 256 (131601 rows, the sum of 456 partials in it), 28 at 100, 13
// at 16; a column at a time took 356 and 90 us at 256 and 100.
constexpr int ST = 512, SB = 32;

// Threads side by side on columns; ST / solve_width share a column's sum.
__host__ __device__ constexpr int solve_width(int n) {
  int w = ST;
  while (w / 2 >= n && w > 32) w >>= 1;
  return w;
}

__global__ void __launch_bounds__(ST) k_lstsq_solve(const double* partial, int64_t nsplit, int n,
                                                    const double* R, int64_t ldr,
                                                    double* x) {
  grid_chain();
  extern __shared__ double c[];  // c[n], then ST partial sums where columns' sums are shared
  double* ps = c + n;
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const int width = solve_width(n), parts = ST / width, part = t / width;
  for (int j0 = 0; j0 < n; j0 += width) {
    const int j = j0 + t % width;
    double s = 0.0;
    if (j < n) {
      int64_t k = part;
      for (; k + 7 * parts < nsplit; k += 8 * parts) {
        double v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) v[u] = partial[(k + u * parts) * n + j];
#pragma unroll
        for (int u = 0; u < 8; ++u) s += v[u];
      }
      for (; k < nsplit; k += parts) s += partial[k * n + j];
    }
    if (parts > 1) {
      ps[t] = s;
      __syncthreads();
      if (part == 0)
        for (int k = 1; k < parts; ++k) s += ps[t + k * width];
    }
    if (part == 0 && j < n) c[j] = s;
  }
  __syncthreads();
  const int last = (n - 1) / SB;  // block of the last columns
  if (warp < 2) {
    double rr[SB];  // this lane's row of the diagonal block, divided by the columns' diagonal entries
    double rinv = 1.0, rd = 1.0;
    bool safe = true;
    auto load_block = [&](int B0) {  // unscaled
#pragma unroll
      for (int k = 0; k < SB; ++k)
        rr[k] = (lane < k && B0 + k < n) ? R[(B0 + lane) + (int64_t)(B0 + k) * ldr] : 0.0;
      rd = B0 + lane < n ? R[(B0 + lane) + (int64_t)(B0 + lane) * ldr] : 1.0;
      rinv = 1.0 / rd;
      const double a = fabs(rd);
      int top = 0;  // high word of the largest entry
#pragma unroll
      for (int k = 0; k < SB; ++k) top = max(top, __double2hiint(rr[k]) & 0x7FFFFFFF);
      safe = __all_sync(0xffffffffu, a > 0x1p-500 && a < 0x1p500 && top < (1023 + 500) << 20);
    };
    // A block's 93 operations for the quotients take 3 us: in three parts, they
    // hide behind an update, the other warp's solve and the update after that
    // (8192 x 256: 2575 us with products, 2593 in one part, 2584 in three).
    constexpr int K1 = 11, K2 = 21;
    auto scale = [&](int B0, auto from, auto to) {
#pragma unroll
      for (int k = decltype(from)::value; k < decltype(to)::value; ++k)
        if (B0 + k < n) rr[k] = rs_quotient(rr[k], __shfl_sync(0xffffffffu, rd, k), __shfl_sync(0xffffffffu, rinv, k));
    };
    using std::integral_constant;
    const integral_constant<int, 1> k0{};
    const integral_constant<int, K1> k1{};
    const integral_constant<int, K2> k2{};
    const integral_constant<int, SB> k3{};
    if (last - warp >= 0) {
      load_block((last - warp) * SB);
      scale((last - warp) * SB, k0, k3);
    }
    for (int blk = last; blk >= 0; --blk) {
      const int B0 = blk * SB;
      const bool mine = ((last - blk) & 1) == warp;
      if (mine) {
        double ci = B0 + lane < n ? c[B0 + lane] : 0.0;
        if (safe) {
#pragma unroll
          for (int k = SB - 1; k >= 1; --k) ci = fma(-rr[k], __shfl_sync(0xffffffffu, ci, k), ci);
          const double q = rs_quotient(ci, rd, rinv);
          ci = isfinite(q) ? q : ci * rinv;
        } else {
#pragma unroll 1
          for (int k = min(SB, n - B0) - 1; k >= 0; --k) {
            if (lane == k) ci = ci / rd;
            const double xk = __shfl_sync(0xffffffffu, ci, k);
            if (lane < k) ci = fma(-R[(B0 + lane) + (int64_t)(B0 + k) * ldr], xk, ci);
          }
        }
        if (B0 + lane < n) {
          c[B0 + lane] = ci;
          x[B0 + lane] = ci;
        }
      } else if (blk >= 1 && blk < last) {
        scale(B0 - SB, k1, k2);
      }
      __syncthreads();
      if (mine) {
        if (blk >= 2) {
          load_block(B0 - 2 * SB);
          scale(B0 - 2 * SB, k0, k1);
        }
      } else if (blk >= 1 && blk < last) {
        scale(B0 - SB, k2, k3);
      }
      __syncthreads();
    }
  } else {
    constexpr int H = SB / 2, PASS = (ST / 32 - 2) * 16;  // rows updated side by side
    const int half = lane >> 4, row = (warp - 2) * 16 + (lane & 15);
    for (int blk = last; blk >= 0; --blk) {
      const int B0 = blk * SB, kh = min(SB, n - B0) - H * half;  // columns of this lane's half
      const double* xb = c + B0 + H * half;
      const double* Rb = R + (int64_t)(B0 + H * half) * ldr;
      double v[H];
#pragma unroll
      for (int k = 0; k < H; ++k) v[k] = ((warp - 2) * 16 < B0 && k < kh) ? Rb[row + (int64_t)k * ldr] : 0.0;
      __syncthreads();
      // a warp's rows are all in or all out (B0 is a multiple of 32), and one that is out issues nothing
      for (int i0 = 0; i0 + (warp - 2) * 16 < B0; i0 += PASS) {
        const int i = i0 + row;
        if (i0 > 0) {
#pragma unroll
          for (int k = 0; k < H; ++k) v[k] = (k < kh) ? Rb[i + (int64_t)k * ldr] : 0.0;
        }
        double s = 0.0;
#pragma unroll
        for (int k = 0; k < H; ++k)
          if (k < kh) s = fma(-v[k], xb[k], s);
        __syncwarp();
        s += __shfl_xor_sync(0xffffffffu, s, 16);
        if (half == 0) c[i] += s;
      }
      __syncthreads();
    }
  }
}

// Column groups side by side in a CTA: a power of two up to its warps.
int gemv_groups(int n) {
  int g = 1;
  while (g < GW && g * GC < n) g *= 2;
  return g;
}

}  // namespace

// Row ranges of at least 128 rows, in one wave of three CTAs per SM (what the
// kernel's registers allow) over all column groups.
int64_t gemv_splits(int64_t m, int n) {
  int dev = 0, sms = 148;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const int gpc = gemv_groups(n);
  const int64_t rs = GW / gpc, gy = ceil_div(n, gpc * GC);
  const int64_t gx = std::max<int64_t>(1, std::min<int64_t>(ceil_div(m, 128 * rs), (int64_t)3 * sms / gy));
  return gx * rs;
}

cudaError_t gemv_t_partials(const double* Q, int64_t ldq, int64_t m, int n, const double* b, int64_t nsplit,
                            double* partial, Lane s) {
  const int gpc = gemv_groups(n);
  const int64_t rows_per = ceil_div(ceil_div(m, nsplit), 32) * 32;  // ranges start on 256-byte lines
  dim3 grid((unsigned)(nsplit / (GW / gpc)), (unsigned)ceil_div(n, gpc * GC));
  cudaError_t e = launch_chained(k_gemv_t_partial, grid, dim3(GT), 0, s, dim3(1),
                                 chain_early((int64_t)grid.x * grid.y), Q, ldq, m, n, b, rows_per, gpc, partial);
  if (e != cudaSuccess) return e;
  count_launch();
  return cudaGetLastError();
}

cudaError_t lstsq_solve(const double* partial, int64_t nsplit, int n, const double* R, int64_t ldr, double* x,
                        Lane s) {
  const size_t sm = ((size_t)n + (solve_width(n) < ST ? ST : 0)) * sizeof(double);
  if (sm > 48 * 1024) {
    cudaError_t e = cudaFuncSetAttribute(k_lstsq_solve, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return e;
  }
  cudaError_t e = launch_chained(k_lstsq_solve, dim3(1), dim3(ST), sm, s, dim3(1), true, partial, nsplit, n,
                                 R, ldr, x);
  if (e != cudaSuccess) return e;
  count_launch();
  return cudaGetLastError();
}

}  // namespace cqr2
