// Q-forming multiply Q = A R^-1 (Algorithm CQR step 3) for n <= 256, and its
// fusion with the next pass's Gram (Algorithm CQR2 steps 1-2: the Q1 panel
// that pass 1 produces is accumulated into pass 2's Gram while it is still on
// chip, so Q1 is not read back from memory for the Gram).
//
// R^-1 is upper triangular, so column j of Q needs only k <= j. One lane
// owns one row of a 32-row panel; a warp owns groups of w = ceil(n / 16)
// adjacent columns, so every lane of a warp runs the same k range and no FP64
// lane is spent on the zero triangle. The ng = ceil(n / w) groups end at column
// n - 1, so the columns a ragged n lacks are missing from the first group,
// whose k range is the shortest, and not from the last, whose is the longest.
// Warp v takes groups v and ng - 1 - v, which evens out the warps' work. (Groups
// of a power of two from column 0 on, as before: at n = 100 the busiest warp
// had 1.5 times the mean.) R^-1 is pre-packed per group ([group][k][c],
// c padded to an even count for 16-byte loads) and read as a warp-wide
// broadcast, with ordinary loads: the kernel may be set up while its
// predecessor still writes R^-1 (grid_chain), and the read-only path is for
// data that no one writes during the kernel's lifetime. The A panel is staged
// in shared memory as [k][row], which makes both the global loads and the
// shared loads conflict-free.
#include <algorithm>

#include "gram_pairs.cuh"
#include "kernels.h"

namespace cqr2 {
namespace {

constexpr int PANEL = QFORM_PANEL;  // rows per panel (one per lane)
constexpr int NGROUP = 16;  // column groups
constexpr int QT = 256;     // threads per CTA

__host__ __device__ constexpr int pitch_of(int w) { return w + (w & 1); }
// Columns missing from the first group.
__host__ __device__ constexpr int lead_of(int n, int w) { return (n + w - 1) / w * w - n; }

__global__ void k_pack_rinv(const double* X, int64_t ldx, int n, int w, bool from_lower,
                            double* Rp) {
  grid_chain();
  const int wp = pitch_of(w), lead = lead_of(n, w);
  const int64_t total = (int64_t)NGROUP * n * wp;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
    const int c = (int)(e % wp);
    const int k = (int)((e / wp) % n);
    const int g = (int)(e / ((int64_t)wp * n));
    const int col = g * w + c - lead;
    double v = 0.0;
    if (c < w && col >= 0 && col < n && k <= col) v = from_lower ? X[col + (int64_t)k * ldx] : X[k + (int64_t)col * ldx];
    Rp[e] = v;
  }
}

template <int W>
__device__ __forceinline__ void load_w(const double* p, double (&r)[W]) {
#pragma unroll
  for (int c = 0; c < W; c += 2) {
    const double2 v = *reinterpret_cast<const double2*>(p + c);
    r[c] = v.x;
    if (c + 1 < W) r[c + 1] = v.y;
  }
}

// Computes the W columns of group g for the lane's row of the staged panel.
template <int W>
__device__ __forceinline__ void qform_group(const double* As, int lane, int n, int g,
                                            const double* Rp, double (&acc)[W]) {
  constexpr int WP = pitch_of(W);
  const int c0 = g * W - lead_of(n, W);  // negative for a ragged first group
  const double* rp = Rp + (int64_t)g * n * WP;
#pragma unroll
  for (int c = 0; c < W; ++c) acc[c] = 0.0;
#pragma unroll 4
  for (int k = 0; k < c0; ++k) {
    const double a = As[k * PANEL + lane];
    double r[W];
    load_w<W>(rp + (int64_t)k * WP, r);
#pragma unroll
    for (int c = 0; c < W; ++c) acc[c] = fma(a, r[c], acc[c]);
  }
#pragma unroll
  for (int kk = 0; kk < W; ++kk) {
    const int k = c0 + kk;
    if (k >= 0) {
      const double a = As[k * PANEL + lane];
      double r[W];
      load_w<W>(rp + (int64_t)k * WP, r);
#pragma unroll
      for (int c = kk; c < W; ++c) acc[c] = fma(a, r[c], acc[c]);
    }
  }
}

__device__ __forceinline__ void stage_panel(const double* A, int64_t lda, int64_t m, int n, int64_t row0,
                                            double* As) {
  for (int e = threadIdx.x; e < n * PANEL; e += QT) {
    const int r = e & (PANEL - 1), k = e >> 5;
    const int64_t row = row0 + r;
    As[e] = row < m ? A[row + (int64_t)k * lda] : 0.0;
  }
}

// A is deliberately not __restrict__: Q may alias A.
template <int W>
__global__ void __launch_bounds__(QT) k_qform_small(const double* A, int64_t lda, int64_t m, int n,
                                                    const double* Rp, double* Q, int64_t ldq,
                                                    int64_t npanels) {
  grid_chain();
  extern __shared__ double As[];  // [n][PANEL]
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int ng = (n + W - 1) / W, lead = lead_of(n, W);
  for (int64_t panel = blockIdx.x; panel < npanels; panel += gridDim.x) {
    const int64_t row0 = panel * PANEL;
    stage_panel(A, lda, m, n, row0, As);
    __syncthreads();
    const int64_t row = row0 + lane;
#pragma unroll 1
    for (int half = 0; half < 2; ++half) {
      const int g = half ? ng - 1 - warp : warp;
      if (half ? g <= warp : 2 * warp > ng - 1) continue;
      double acc[W];
      qform_group<W>(As, lane, n, g, Rp, acc);
      if (row < m) {
#pragma unroll
        for (int c = 0; c < W; ++c)
          if (g * W + c >= lead) Q[row + (int64_t)(g * W + c - lead) * ldq] = acc[c];
      }
    }
    __syncthreads();
  }
}

// Fused Q-form + Gram for n <= 128 (one diagonal Gram tile), MAXS >=
// gram_slots(n). The Gram part reads the freshly formed Q panel from shared
// memory ([row][col], odd pitch).
template <int W, int MAXS>
__global__ void __launch_bounds__(QT) k_qform_gram_small(const double* A, int64_t lda, int64_t m, int n,
                                                         const double* Rp, double* Q, int64_t ldq,
                                                         int64_t rows_per_split, int T, double* partial) {
  grid_chain();
  static_assert(QT == GRAM_NT, "the pair list is dealt to this block's threads");
  extern __shared__ double smem[];
  const int pitch = n | 1, ng = (n + W - 1) / W, lead = lead_of(n, W);
  double* As = smem;                       // [n][PANEL]
  double* Qs = smem + (size_t)n * PANEL;   // [PANEL][pitch]
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  GramPairs<MAXS> pairs;
  pairs.init(t, n);

  const int64_t r_begin = (int64_t)blockIdx.x * rows_per_split;
  const int64_t r_end = min(m, r_begin + rows_per_split);
  for (int64_t row0 = r_begin; row0 < r_end; row0 += PANEL) {
    stage_panel(A, lda, r_end, n, row0, As);
    __syncthreads();
    const int64_t row = row0 + lane;
#pragma unroll 1
    for (int half = 0; half < 2; ++half) {
      const int g = half ? ng - 1 - warp : warp;
      if (half ? g <= warp : 2 * warp > ng - 1) continue;
      double acc[W];
      qform_group<W>(As, lane, n, g, Rp, acc);
#pragma unroll
      for (int c = 0; c < W; ++c) {
        const int col = g * W + c - lead;
        if (col >= 0) {
          Qs[lane * pitch + col] = acc[c];
          if (row < r_end) Q[row + (int64_t)col * ldq] = acc[c];
        }
      }
    }
    __syncthreads();
    pairs.add(Qs, pitch, PANEL);
    __syncthreads();
  }
  pairs.store(partial + (int64_t)blockIdx.x * (T * T), T);
}

int sm_count() {
  int dev = 0, sms = 148;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  return sms;
}

// A grid that is set up early asks for more than half of an SM's shared memory,
// so that no two of its CTAs share an SM: placed while the predecessor still
// holds most SMs, they piled up on the others, up to three on one, each with a
// panel of 70 (n = 128) to 277 us (n = 256). us per factorization: 2432 x 256
// 2407 -> 1382, 512 x 256 2207 -> 1183, 2000 x 200 1399 -> 928; 1024 x 16 and
// 4096 x 64 unchanged.
constexpr int QFORM_ALONE_SMEM = 118 * 1024;
static_assert(QFORM_ALONE_SMEM >= 256 * PANEL * (int)sizeof(double), "the widest matrix's panel");

template <int W>
cudaError_t launch_qform(const double* A, int64_t lda, int64_t m, int n, const double* Rp, double* Q, int64_t ldq,
                         Lane s) {
  const size_t sm = (size_t)n * PANEL * sizeof(double);
  auto kern = k_qform_small<W>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, QFORM_ALONE_SMEM);
  if (e != cudaSuccess) return e;
  const int64_t npanels = ceil_div(m, PANEL);
  int per_sm = 1;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, QT, sm);
  const int64_t waves = s.shared ? 4 : 1;
  const int64_t grid = std::max<int64_t>(1, std::min<int64_t>(npanels, waves * sm_count() * std::max(1, per_sm)));
  const bool early = chain_early(2 * grid) && !s.shared;
  e = launch_chained(kern, dim3((unsigned)grid), dim3(QT), early ? (size_t)QFORM_ALONE_SMEM : sm, s, dim3(1), early, A,
                     lda, m, n, Rp, Q, ldq, npanels);
  if (e != cudaSuccess) return e;
  count_launch();
  return cudaGetLastError();
}

template <int W, int MAXS>
cudaError_t launch_fused(const double* A, int64_t lda, int64_t m, int n, const double* Rp, double* Q, int64_t ldq,
                         const GramGeom& g, double* partial, Lane s) {
  static_assert(MAXS >= gram_slots(16 * W > 128 ? 128 : 16 * W), "slots of the widest matrix of this group width");
  const size_t sm = ((size_t)n * PANEL + (size_t)PANEL * (n | 1)) * sizeof(double);
  auto kern = k_qform_gram_small<W, MAXS>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)((128 + 129) * PANEL * sizeof(double)));
  if (e != cudaSuccess) return e;
  e = launch_chained(kern, dim3((unsigned)g.nsplit), dim3(QT), sm, s, dim3(1), chain_early(2 * g.nsplit), A, lda, m,
                     n, Rp, Q, ldq, g.rows_per_split, g.T, partial);
  if (e != cudaSuccess) return e;
  count_launch();
  return cudaGetLastError();
}

}  // namespace

int qform_group_width(int n) { return n > 256 ? 0 : (int)ceil_div(n, NGROUP); }

size_t rpack_doubles(int n) {
  const int w = qform_group_width(n);
  return (size_t)NGROUP * n * (w ? pitch_of(w) : 0);
}

static cudaError_t pack(const double* X, int64_t ldx, int n, bool lower, double* Rp, Lane s) {
  const int w = qform_group_width(n);
  if (!w) return cudaErrorInvalidValue;
  const int64_t total = (int64_t)rpack_doubles(n);
  const int grid = (int)std::min<int64_t>(ceil_div(total, 256), 4096);
  cudaError_t e = launch_chained(k_pack_rinv, dim3((unsigned)grid), dim3(256), 0, s, dim3(1), true, X, ldx, n, w,
                                 lower, Rp);
  if (e != cudaSuccess) return e;
  count_launch();
  return cudaGetLastError();
}

cudaError_t pack_rinv_from_lower(const double* Y, int64_t ldy, int n, double* Rp, Lane s) {
  return pack(Y, ldy, n, true, Rp, s);
}

cudaError_t pack_rinv_from_upper(const double* Rinv, int64_t ld, int n, double* Rp, Lane s) {
  return pack(Rinv, ld, n, false, Rp, s);
}

cudaError_t qform_small(const double* A, int64_t lda, int64_t m, int n, const double* Rp, double* Q, int64_t ldq,
                        Lane s) {
  switch (qform_group_width(n)) {
    case 1: return launch_qform<1>(A, lda, m, n, Rp, Q, ldq, s);
    case 2: return launch_qform<2>(A, lda, m, n, Rp, Q, ldq, s);
    case 3: return launch_qform<3>(A, lda, m, n, Rp, Q, ldq, s);
    case 4: return launch_qform<4>(A, lda, m, n, Rp, Q, ldq, s);
    case 5: return launch_qform<5>(A, lda, m, n, Rp, Q, ldq, s);
    case 6: return launch_qform<6>(A, lda, m, n, Rp, Q, ldq, s);
    case 7: return launch_qform<7>(A, lda, m, n, Rp, Q, ldq, s);
    case 8: return launch_qform<8>(A, lda, m, n, Rp, Q, ldq, s);
    case 9: return launch_qform<9>(A, lda, m, n, Rp, Q, ldq, s);
    case 10: return launch_qform<10>(A, lda, m, n, Rp, Q, ldq, s);
    case 11: return launch_qform<11>(A, lda, m, n, Rp, Q, ldq, s);
    case 12: return launch_qform<12>(A, lda, m, n, Rp, Q, ldq, s);
    case 13: return launch_qform<13>(A, lda, m, n, Rp, Q, ldq, s);
    case 14: return launch_qform<14>(A, lda, m, n, Rp, Q, ldq, s);
    case 15: return launch_qform<15>(A, lda, m, n, Rp, Q, ldq, s);
    case 16: return launch_qform<16>(A, lda, m, n, Rp, Q, ldq, s);
    default: return cudaErrorInvalidValue;
  }
}

bool qform_gram_fusable(int n) { return n >= 1 && n <= 128; }

cudaError_t qform_gram_small(const double* A, int64_t lda, int64_t m, int n, const double* Rp, double* Q,
                             int64_t ldq, const GramGeom& g, double* partial, Lane s) {
  if (!qform_gram_fusable(n) || g.ntile != 1 || g.T < n) return cudaErrorInvalidValue;
  switch (qform_group_width(n)) {
    case 1: return launch_fused<1, 8>(A, lda, m, n, Rp, Q, ldq, g, partial, s);
    case 2: return launch_fused<2, 8>(A, lda, m, n, Rp, Q, ldq, g, partial, s);
    case 3: return launch_fused<3, 8>(A, lda, m, n, Rp, Q, ldq, g, partial, s);
    case 4: return launch_fused<4, 16>(A, lda, m, n, Rp, Q, ldq, g, partial, s);
    case 5: return launch_fused<5, 16>(A, lda, m, n, Rp, Q, ldq, g, partial, s);
    case 6: return launch_fused<6, 24>(A, lda, m, n, Rp, Q, ldq, g, partial, s);
    case 7: return launch_fused<7, 33>(A, lda, m, n, Rp, Q, ldq, g, partial, s);
    case 8: return launch_fused<8, 33>(A, lda, m, n, Rp, Q, ldq, g, partial, s);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace cqr2
