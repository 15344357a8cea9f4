// General FP64 GEMM C = alpha op(A) op(B) + beta C (the MM of Section II-A)
// with triangular-structure flags, used for the CholInv recursion
// (Algorithm 1), R = R2 R1, and the Q-forming multiply when n > 256.
//
// T x T x 16 tiles (T = 64 with 256 threads, T = 32 with 128), register
// micro-tiles of 4 rows by T / 16 columns, register double buffering of the
// next k-slice. GB300's FP64 pipe (about 2 FMA per clock per SM) is the bound,
// so the zeros matter more than the load path: a tile's k range is clipped to
// the blocks that the triangles of op(A) and op(B) leave nonzero, within the
// clipped range and in the ragged last tiles a warp skips the 16-column and
// T/4-row groups that hold only zeros or lie outside C, output tiles outside
// the requested triangle are skipped, and elements inside the zero triangle
// are never read (they are masked to zero at load), so callers may leave
// garbage there.
//
// A product with few tiles, or a number of tiles that leaves the last wave
// nearly empty, splits k over up to 8 CTAs per tile. Those form a cluster: each
// leaves its partial tile in its own shared memory and then sums a share of
// the tile's elements over the cluster in split order (deterministic), so no
// scratch and no second launch are needed. With 64 x 64 tiles only, partial
// sums in scratch and no group skipping: CholInv at n = 256 318 us, now 280;
// Q = A R^-1 for 6001 x 777 3.99 ms, now 3.04 (2.9 at the pipe's peak); the
// projections of an 8192 x 2048 factorization on panels of 512 58.8 ms, now
// 44 (43 at the peak); R2 R1 at n = 777 0.80 ms, now 0.22.
#include <algorithm>

#include "kernels.h"

namespace cqr2 {
namespace {

constexpr int BK = 16;

__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ double ld_remote(const double* p, uint32_t rank) {
  uint32_t a;
  double v;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"(rank));
  asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(a) : "memory");
  return v;
}

template <int T, bool TA, bool TB>
__global__ void __launch_bounds__(4 * T) k_gemm_f64(int64_t M, int64_t N, int64_t K, double alpha,
                                                    const double* A, int64_t lda,
                                                    const double* B, int64_t ldb, double beta,
                                                    double* C, int64_t ldc, unsigned flags, int ksplit) {
  grid_chain();
  constexpr int NT = 4 * T, TX = T / 4, NC = T / 16, PITCH = T + 1, NQ = 4;
  static_assert(T * BK / NT == NQ, "elements per thread of a staged slice");
  __shared__ double smem[4 * BK * PITCH];
  double(*As)[BK][PITCH] = reinterpret_cast<double(*)[BK][PITCH]>(smem);
  double(*Bs)[BK][PITCH] = reinterpret_cast<double(*)[BK][PITCH]>(smem + 2 * BK * PITCH);
  // the tiles with the longest k ranges first
  const int64_t bx = (flags & GEMM_A_LOWER) ? gridDim.x - 1 - blockIdx.x : blockIdx.x;
  const int64_t by = (flags & GEMM_B_UPPER) ? gridDim.y - 1 - blockIdx.y : blockIdx.y;
  const int64_t i0 = bx * T, j0 = by * T;
  const int t = threadIdx.x, tx = t % TX, ty = t / TX;

  // (a cluster's CTAs share the tile, so they return together)
  if ((flags & GEMM_C_LOWER) && j0 > i0 + T - 1) return;
  if ((flags & GEMM_C_UPPER) && i0 > j0 + T - 1) {
    if (blockIdx.z > 0) return;
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        const int64_t gi = i0 + tx + TX * r, gj = j0 + ty + 16 * c;
        if (gi < M && gj < N) C[gi + gj * ldc] = 0.0;
      }
    return;
  }
  int64_t kb = 0, ke = K;
  if (flags & GEMM_A_LOWER) ke = min(ke, i0 + T);
  if (flags & GEMM_A_UPPER) kb = max(kb, i0);
  if (flags & GEMM_B_LOWER) kb = max(kb, j0);
  if (flags & GEMM_B_UPPER) ke = min(ke, j0 + T);
  kb = (kb / BK) * BK;
  if (ksplit > 1) {  // this CTA's share of the k range, in whole k-slices
    const int64_t per = ((ke - kb + BK - 1) / BK + ksplit - 1) / ksplit * BK;
    const int64_t z0 = kb + (int64_t)blockIdx.z * per;
    ke = min(ke, z0 + per);
    kb = z0;
  }

  double acc[4][NC];
#pragma unroll
  for (int r = 0; r < 4; ++r)
#pragma unroll
    for (int c = 0; c < NC; ++c) acc[r][c] = 0.0;

  double ra[NQ], rb[NQ];
  auto load = [&](int64_t k0) {
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
      const int e = t + q * NT;
      int i, k;
      if (!TA) { i = e % T; k = e / T; } else { k = e % BK; i = e / BK; }
      const int64_t gi = i0 + i, gk = k0 + k;
      bool ok = gi < M && gk < K;
      if (flags & GEMM_A_LOWER) ok = ok && gk <= gi;
      if (flags & GEMM_A_UPPER) ok = ok && gk >= gi;
      ra[q] = ok ? (TA ? A[gk + gi * lda] : A[gi + gk * lda]) : 0.0;
    }
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
      const int e = t + q * NT;
      int j, k;
      if (!TB) { k = e % BK; j = e / BK; } else { j = e % T; k = e / T; }
      const int64_t gj = j0 + j, gk = k0 + k;
      bool ok = gj < N && gk < K;
      if (flags & GEMM_B_LOWER) ok = ok && gk >= gj;
      if (flags & GEMM_B_UPPER) ok = ok && gk <= gj;
      rb[q] = ok ? (TB ? B[gj + gk * ldb] : B[gk + gj * ldb]) : 0.0;
    }
  };
  auto store = [&](int buf) {
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
      const int e = t + q * NT;
      int i, k;
      if (!TA) { i = e % T; k = e / T; } else { k = e % BK; i = e / BK; }
      As[buf][k][i] = ra[q];
    }
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
      const int e = t + q * NT;
      int j, k;
      if (!TB) { k = e % BK; j = e / BK; } else { j = e % T; k = e / T; }
      Bs[buf][k][j] = rb[q];
    }
  };

  // row groups (TX rows) and column groups (16 columns) inside C
  const int rM = (int)min((int64_t)4, (M - i0 + TX - 1) / TX), cN = (int)min((int64_t)NC, (N - j0 + 15) / 16);
  if (kb < ke) {
    load(kb);
    store(0);
    __syncthreads();
    int buf = 0;
    for (int64_t k0 = kb; k0 < ke; k0 += BK) {
      const bool more = k0 + BK < ke;
      if (more) load(k0 + BK);
      // groups with a nonzero factor in this slice
      int r0 = 0, r1 = rM, c0 = 0, c1 = cN;
      if (flags & GEMM_A_LOWER) r0 = (int)max((int64_t)0, (k0 - i0) / TX);
      if (flags & GEMM_A_UPPER) r1 = (int)min((int64_t)r1, (k0 + BK - 1 - i0) / TX + 1);
      if (flags & GEMM_B_LOWER) c1 = (int)min((int64_t)c1, (k0 + BK - 1 - j0) / 16 + 1);
      if (flags & GEMM_B_UPPER) c0 = (int)max((int64_t)0, (k0 - j0) / 16);
      if (r0 == 0 && r1 == 4 && c0 == 0 && c1 == NC) {
#pragma unroll
        for (int k = 0; k < BK; ++k) {
          double a[4], b[NC];
#pragma unroll
          for (int r = 0; r < 4; ++r) a[r] = As[buf][k][tx + TX * r];
#pragma unroll
          for (int c = 0; c < NC; ++c) b[c] = Bs[buf][k][ty + 16 * c];
#pragma unroll
          for (int r = 0; r < 4; ++r)
#pragma unroll
            for (int c = 0; c < NC; ++c) acc[r][c] = fma(a[r], b[c], acc[r][c]);
        }
      } else {
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
          for (int c = 0; c < NC; ++c)
            if (r >= r0 && r < r1 && c >= c0 && c < c1) {
              double v = acc[r][c];
#pragma unroll 4
              for (int k = 0; k < BK; ++k) v = fma(As[buf][k][tx + TX * r], Bs[buf][k][ty + 16 * c], v);
              acc[r][c] = v;
            }
      }
      if (more) store(buf ^ 1);
      __syncthreads();
      buf ^= 1;
    }
  }

  auto write = [&](int64_t gi, int64_t gj, double v) {
    if (gi >= M || gj >= N) return;
    if ((flags & GEMM_C_LOWER) && gi < gj) return;
    if ((flags & GEMM_C_UPPER) && gi > gj) {
      C[gi + gj * ldc] = 0.0;
      return;
    }
    if (!(flags & GEMM_BETA0)) v = fma(beta, C[gi + gj * ldc], v);
    C[gi + gj * ldc] = v;
  };
  if (ksplit > 1) {
    // this split's partial tile, alpha * sum over its k range, as smem[j T + i]
    static_assert(4 * BK * PITCH >= T * T, "the staging buffers hold a tile");
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
      for (int c = 0; c < NC; ++c) smem[(ty + 16 * c) * T + tx + TX * r] = alpha * acc[r][c];
    cluster_sync();
    const int per = T * T / ksplit;  // ksplit is 2, 4 or 8
    for (int e = (int)blockIdx.z * per + t; e < ((int)blockIdx.z + 1) * per; e += NT) {
      double p[8];
#pragma unroll
      for (int z = 0; z < 8; ++z) p[z] = z < ksplit ? ld_remote(smem + e, z) : 0.0;
      double v = p[0];
      for (int z = 1; z < 8; ++z)
        if (z < ksplit) v += p[z];
      write(i0 + e % T, j0 + e / T, v);
    }
    cluster_sync();  // a CTA's partials stay until everyone has read them
    return;
  }
#pragma unroll
  for (int r = 0; r < 4; ++r)
#pragma unroll
    for (int c = 0; c < NC; ++c) write(i0 + tx + TX * r, j0 + ty + 16 * c, alpha * acc[r][c]);
}

template <int T, bool TA, bool TB>
cudaError_t launch_gemm(int64_t M, int64_t N, int64_t K, double alpha, const double* A, int64_t lda, const double* B,
                        int64_t ldb, double beta, double* C, int64_t ldc, unsigned flags, int ks, Lane s) {
  const dim3 grid((unsigned)ceil_div(M, T), (unsigned)ceil_div(N, T), (unsigned)ks);
  cudaError_t e = launch_chained(k_gemm_f64<T, TA, TB>, grid, dim3(4 * T), 0, s, dim3(1, 1, (unsigned)ks),
                                 chain_early((int64_t)grid.x * grid.y * grid.z), M, N, K, alpha, A, lda, B, ldb, beta, C,
                                 ldc, flags, ks);
  if (e != cudaSuccess) return e;
  count_launch();
  return cudaGetLastError();
}

template <int T>
cudaError_t launch_gemm_t(int64_t M, int64_t N, int64_t K, double alpha, const double* A, int64_t lda, const double* B,
                          int64_t ldb, double beta, double* C, int64_t ldc, unsigned flags, int ks, Lane s) {
  const bool ta = flags & GEMM_TA, tb = flags & GEMM_TB;
  if (!ta && !tb) return launch_gemm<T, false, false>(M, N, K, alpha, A, lda, B, ldb, beta, C, ldc, flags, ks, s);
  if (!ta && tb) return launch_gemm<T, false, true>(M, N, K, alpha, A, lda, B, ldb, beta, C, ldc, flags, ks, s);
  if (ta && !tb) return launch_gemm<T, true, false>(M, N, K, alpha, A, lda, B, ldb, beta, C, ldc, flags, ks, s);
  return launch_gemm<T, true, true>(M, N, K, alpha, A, lda, B, ldb, beta, C, ldc, flags, ks, s);
}

// Tile size and k split from a model of the time in FP64 slots of one SM (a
// warp instruction, 16 clocks): the SM with the most CTAs does
// ceil(tiles ks / SMs) shares of T^2 k / 32 / ks slots, where k is the mean
// range over the tiles with work, and no less than one CTA's longest range;
// each CTA also costs about 120 slots to fill and drain (1 us), a cluster's
// sum 60 more. Ties go to the larger tile and the smaller split.
void gemm_shape(int64_t M, int64_t N, int64_t K, unsigned flags, int sms, int max_split, int* T, int* ks) {
  double best = 0.0;
  const bool tri_k = flags & (GEMM_A_LOWER | GEMM_A_UPPER | GEMM_B_LOWER | GEMM_B_UPPER);
  const bool tri_c = flags & (GEMM_C_LOWER | GEMM_C_UPPER);
  for (int t = 64; t >= 32; t /= 2) {
    const double gx = (double)ceil_div(M, t), gy = (double)ceil_div(N, t);
    const double tiles = tri_c ? std::max(1.0, 0.5 * gx * gy + 0.5 * std::min(gx, gy)) : gx * gy;
    const double kmean = tri_k ? std::min((double)K, 0.5 * (double)K + 0.5 * t) : (double)K;
    for (int z = 1; z <= max_split; z *= 2) {
      if (z > 1 && K < BK * z) break;
      const double cta = t * t / 32.0 / z;
      const double fixed = 120.0 + (z > 1 ? 60.0 : 0.0);
      const double shares = std::ceil(tiles * z / sms);
      const double est = std::max(shares * (cta * kmean + (shares > 3 ? fixed / 3 : fixed)), cta * (double)K + fixed);
      if (best == 0.0 || est < 0.97 * best) {
        best = est;
        *T = t;
        *ks = z;
      }
    }
  }
}

}  // namespace

cudaError_t gemm_f64(int64_t M, int64_t N, int64_t K, double alpha, const double* A, int64_t lda, const double* B,
                     int64_t ldb, double beta, double* C, int64_t ldc, unsigned flags, Lane s) {
  if (M <= 0 || N <= 0) return cudaSuccess;
  int sms = 148, dev = 0, T = 64, ks = 1;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  gemm_shape(M, N, K, flags, sms, s.shared ? 1 : 8, &T, &ks);
  if (ceil_div(N, T) > 65535) return cudaErrorInvalidValue;
  return T == 64 ? launch_gemm_t<64>(M, N, K, alpha, A, lda, B, ldb, beta, C, ldc, flags, ks, s)
                 : launch_gemm_t<32>(M, N, K, alpha, A, lda, B, ldb, beta, C, ldc, flags, ks, s);
}

// R = op(A) B of two upper-triangular n x n factors (the R2 R1 of Algorithm
// CQR2), n <= TRMM_SMALL_MAX, in one launch: CTA j forms column j; four
// threads share each element, thread q summing op(A)(i, k) B(k, j) over
// k = i + q, i + q + 4, ... <= j in order, and the four partial sums are
// added in a fixed order through two shuffles (a chain of at most 32 FMAs
// where one thread per element would hold 128). C below the diagonal is
// written as 0. op(A)(i, k) = A(k, i) when a_trans (A holds the lower
// transpose, as the Cholesky factor L2 does), else A(i, k). The general GEMM
// has at most 16 tiles for this 2 n^3 / 6 flop product and stages each in shared
// memory: 1024 x 32 takes 73 us with this kernel and 79 with the GEMM, 1024 x 128
// 410 and 416.
constexpr int TRMM_PARTS = 4;
__global__ void __launch_bounds__(TRMM_PARTS * TRMM_SMALL_MAX)
    k_trmm_upper_small(int n, const double* A, int64_t lda, bool a_trans, const double* B,
                       int64_t ldb, double* C, int64_t ldc) {
  grid_chain();
  __shared__ double bj[TRMM_SMALL_MAX];
  const int j = blockIdx.x, t = threadIdx.x, i = t / TRMM_PARTS, q = t % TRMM_PARTS;
  for (int k = t; k <= j; k += blockDim.x) bj[k] = B[k + (int64_t)j * ldb];
  __syncthreads();
  double acc = 0.0;
  if (i <= j) {  // i < n since j < n
    if (a_trans) {
      const double* a = A + (int64_t)i * lda;  // column i of the lower factor
#pragma unroll 4
      for (int k = i + q; k <= j; k += TRMM_PARTS) acc = fma(a[k], bj[k], acc);
    } else {
#pragma unroll 4
      for (int k = i + q; k <= j; k += TRMM_PARTS) acc = fma(A[i + (int64_t)k * lda], bj[k], acc);
    }
  }
  // (p0 + p1) + (p2 + p3): the four threads of an element are adjacent lanes
  acc += __shfl_xor_sync(0xffffffffu, acc, 1);
  acc += __shfl_xor_sync(0xffffffffu, acc, 2);
  if (q == 0 && i < n) C[i + (int64_t)j * ldc] = acc;
}

cudaError_t trmm_upper_small(int n, const double* A, int64_t lda, bool a_trans, const double* B, int64_t ldb,
                             double* C, int64_t ldc, Lane s) {
  if (n < 1 || n > TRMM_SMALL_MAX) return cudaErrorInvalidValue;
  const int threads = (TRMM_PARTS * n + 31) / 32 * 32;
  cudaError_t e = launch_chained(k_trmm_upper_small, dim3((unsigned)n), dim3((unsigned)threads), 0, s, dim3(1), true,
                                 n, A, lda, a_trans, B, ldb, C, ldc);
  if (e != cudaSuccess) return e;
  count_launch();
  return cudaGetLastError();
}

}  // namespace cqr2
