// Split-m Gram (Syrk, Section II-A; Algorithm CQR step 1): W = A^T A.
//
// The n x n upper triangle is cut into T x T tiles (diagonal and strictly
// upper), T at most 128 and chosen so that the tiles are nearly equal (the
// last ones narrower). A CTA owns one range of rows of A and one off-diagonal
// tile or two diagonal ones (about the same work) and accumulates the range's
// partial tiles in registers; a second kernel sums the ranges' partials in a
// fixed order (deterministic), which is the one-GPU counterpart of the 1D
// algorithm's local Syrk + Allreduce (Algorithm 1D-CQR).
//
// GB300 FP64 runs at about 2 FMA per clock per SM and a warp instruction pays
// for all 32 lanes whether or not they are active, so no slot is spent on
// padding: diagonal tiles use the flattened list of their upper pairs
// (gram_pairs.cuh), off-diagonal tiles give each lane one column of the first
// block (T is a multiple of 16, so two lanes per column fill whole warps) and
// every second row of the other (a shared-memory broadcast), and the row
// ranges are cut so that the CTAs, all of equal work, fill whole waves.
// Row panels of KC rows are staged through double-buffered shared memory with
// cp.async; the layout [row][column] (odd pitch) makes the copies' lanes, which
// differ in the row, hit distinct banks.
#include <algorithm>
#include <mutex>

#include "../../include/cqr2.h"
#include "gram_pairs.cuh"
#include "kernels.h"

namespace cqr2 {
namespace {

constexpr int KC = 32;  // rows per staged chunk

// Scratch of the allocation-free Gram entry point (cqr2_syrk_noalloc): the
// split-m partial tiles live in this fixed device array instead of a plan's
// workspace. It belongs to this file's module: a device holds it from the
// first time the module is loaded there (the first Gram kernel or
// cqr2_syrk_noalloc call on that device, under CUDA's default lazy loading)
// until the process exits.
constexpr size_t NOALLOC_DOUBLES = CQR2_NOALLOC_SCRATCH_BYTES / sizeof(double);
static __device__ __align__(256) double g_noalloc_scratch[NOALLOC_DOUBLES];

constexpr int NT = GRAM_NT;

// Rows [r0, r1) of columns c0 .. c0 + w - 1 into X[row][column], zeros past r1.
__device__ __forceinline__ void load_chunk(const double* A, int64_t lda, int64_t r0, int64_t r1, int c0, int w, double* X,
                                           int pitch) {
  const int kk = threadIdx.x % KC;
  const int64_t row = r0 + kk;
  const bool ok = row < r1;
  const double* src = A + (ok ? row : 0) + (int64_t)c0 * lda;
#pragma unroll 4
  for (int c = threadIdx.x / KC; c < w; c += NT / KC) cp_async8(X + kk * pitch + c, src + (int64_t)c * lda, ok ? 8 : 0);
}

// One diagonal tile of width w at column c0 over rows [r0, r1).
template <int MAXS>
__device__ __forceinline__ void diag_item(const double* A, int64_t lda, int64_t r0, int64_t r1, int c0, int w,
                                          double* smem, double* out, int T) {
  const int pitch = w | 1;
  GramPairs<MAXS> pairs;
  pairs.init(threadIdx.x, w);
  double* cur = smem;
  double* nxt = smem + KC * pitch;
  load_chunk(A, lda, r0, r1, c0, w, cur, pitch);
  cp_async_commit();
  for (int64_t r = r0; r < r1; r += KC) {
    if (r + KC < r1) load_chunk(A, lda, r + KC, r1, c0, w, nxt, pitch);
    cp_async_commit();
    cp_async_wait<1>();
    __syncthreads();
    pairs.add(cur, pitch, (int)min((int64_t)KC, (r1 - r + 3) & ~(int64_t)3));
    __syncthreads();
    double* x = cur;
    cur = nxt;
    nxt = x;
  }
  pairs.store(out, T);
}

// The off-diagonal tile of columns cI .. cI + T - 1 and cJ .. cJ + wJ - 1
// (wJ <= T) over rows [r0, r1): lane column i = t % T of the first block,
// columns t / T, t / T + 2, ... of the second.
template <int S>
__device__ __forceinline__ void off_item(const double* A, int64_t lda, int64_t r0, int64_t r1, int cI, int cJ,
                                         int wJ, double* smem, double* out, int T) {
  const int t = threadIdx.x, pitch = T | 1, i = t % T, jh = t / T;
  const bool live = jh < 2;  // whole warps: T is a multiple of 16
  double acc[S];
#pragma unroll
  for (int s = 0; s < S; ++s) acc[s] = 0.0;
  double* cur = smem;
  double* nxt = smem + 2 * KC * pitch;
  load_chunk(A, lda, r0, r1, cI, T, cur, pitch);
  load_chunk(A, lda, r0, r1, cJ, wJ, cur + KC * pitch, pitch);
  cp_async_commit();
  for (int64_t r = r0; r < r1; r += KC) {
    if (r + KC < r1) {
      load_chunk(A, lda, r + KC, r1, cI, T, nxt, pitch);
      load_chunk(A, lda, r + KC, r1, cJ, wJ, nxt + KC * pitch, pitch);
    }
    cp_async_commit();
    cp_async_wait<1>();
    __syncthreads();
    if (live) {
      const int rows = (int)min((int64_t)KC, (r1 - r + 3) & ~(int64_t)3);
      const double* X = cur + i;
      const double* Y = cur + KC * pitch + jh;
      for (int k = 0; k < rows; k += 4)
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const double x = X[(k + u) * pitch];
          const double* y = Y + (k + u) * pitch;
          // columns past wJ read stale staging words; they are not stored
#pragma unroll
          for (int s = 0; s < S; ++s) acc[s] = fma(x, y[2 * s], acc[s]);
        }
    }
    __syncthreads();
    double* x = cur;
    cur = nxt;
    nxt = x;
  }
  if (live)
#pragma unroll
    for (int s = 0; s < S; ++s)
      if (jh + 2 * s < wJ) out[i + (jh + 2 * s) * T] = acc[s];
}

// One diagonal tile (n <= 128) of at most MAXS slots per thread.
template <int MAXS>
__global__ void __launch_bounds__(NT, MAXS <= 8 ? 3 : (MAXS <= 16 ? 2 : 1))
    k_gram_diag(const double* A, int64_t lda, int64_t m, int n, int64_t rows_per_split, int T,
                double* partial) {
  grid_chain();
  extern __shared__ double smem[];
  const int64_t r0 = (int64_t)blockIdx.x * rows_per_split, r1 = min(m, r0 + rows_per_split);
  diag_item<MAXS>(A, lda, r0, r1, 0, n, smem, partial + (int64_t)blockIdx.x * T * T, T);
}

// Several tiles: blockIdx.y < noff takes an off-diagonal tile, the others two
// diagonal ones in turn.
__global__ void __launch_bounds__(NT, 1)
    k_gram_tiles(const double* A, int64_t lda, int64_t m, int n, int64_t rows_per_split, int T, int ntile,
                 int ntiles_total, double* partial) {
  extern __shared__ double smem[];
  const int64_t r0 = (int64_t)blockIdx.x * rows_per_split, r1 = min(m, r0 + rows_per_split);
  double* out = partial + (int64_t)blockIdx.x * ntiles_total * (int64_t)(T * T);
  const int noff = ntiles_total - ntile;
  if ((int)blockIdx.y < noff) {
    int rem = blockIdx.y, I = 0;
    while (rem >= ntile - 1 - I) {
      rem -= ntile - 1 - I;
      ++I;
    }
    const int J = I + 1 + rem, wJ = min(T, n - J * T);
    double* o = out + (int64_t)(ntile + blockIdx.y) * (T * T);
    // accumulators for 16, 32, ... columns of the narrower last block
    switch ((wJ + 15) / 16) {
      case 1: off_item<8>(A, lda, r0, r1, I * T, J * T, wJ, smem, o, T); break;
      case 2: off_item<16>(A, lda, r0, r1, I * T, J * T, wJ, smem, o, T); break;
      case 3: off_item<24>(A, lda, r0, r1, I * T, J * T, wJ, smem, o, T); break;
      case 4: off_item<32>(A, lda, r0, r1, I * T, J * T, wJ, smem, o, T); break;
      case 5: off_item<40>(A, lda, r0, r1, I * T, J * T, wJ, smem, o, T); break;
      case 6: off_item<48>(A, lda, r0, r1, I * T, J * T, wJ, smem, o, T); break;
      case 7: off_item<56>(A, lda, r0, r1, I * T, J * T, wJ, smem, o, T); break;
      default: off_item<64>(A, lda, r0, r1, I * T, J * T, wJ, smem, o, T); break;
    }
    return;
  }
  const int d0 = 2 * ((int)blockIdx.y - noff);
  for (int d = d0; d < min(d0 + 2, ntile); ++d) {
    const int w = min(T, n - d * T);
    __syncthreads();
    diag_item<gram_slots(128)>(A, lda, r0, r1, d * T, w, smem, out + (int64_t)d * (T * T), T);
  }
}

// W = the sum of the row ranges' partial tiles, mirrored. The ranges are cut
// into RC contiguous chunks: warp c of a block sums chunk c for 32 elements
// of one column, in range order, and thread c = 0 adds the chunk sums in
// chunk order -- the same fixed order on every call (deterministic), with RC
// warps sharing each element's long sum (the FP64 pipe charges every warp
// instruction in full, so one thread per element and hundreds of ranges left
// most of the GPU idle).
constexpr int GRAM_RC = 8;
__global__ void __launch_bounds__(32 * GRAM_RC) k_gram_reduce(const double* partial, int64_t nsplit,
                                                              int T, int ntile, int ntiles_total, int n,
                                                              double* W, int64_t ldw) {
  grid_chain();
  __shared__ double part[GRAM_RC][32];
  const int lane = threadIdx.x & 31, c = threadIdx.x >> 5;
  const int i = blockIdx.x * 32 + lane;
  const int j = blockIdx.y;
  const bool live = i < n && i <= j;
  double s = 0.0;
  if (live) {
    const int I = i / T, Jt = j / T;
    const int tile = I == Jt ? I : ntile + I * ntile - I * (I + 1) / 2 + (Jt - I - 1);
    const int64_t loc = (i - I * T) + (int64_t)(j - Jt * T) * T;
    const int64_t stride = (int64_t)ntiles_total * T * T;
    const double* p = partial + (int64_t)tile * T * T + loc;
    const int64_t b0 = nsplit * c / GRAM_RC, b1 = nsplit * (c + 1) / GRAM_RC;
    int64_t b = b0;
    for (; b + 8 <= b1; b += 8) {  // eight loads in flight
      double v[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) v[u] = p[(b + u) * stride];
#pragma unroll
      for (int u = 0; u < 8; ++u) s += v[u];
    }
    for (; b < b1; ++b) s += p[b * stride];
  }
  part[c][lane] = s;
  __syncthreads();
  if (c == 0 && live) {
    double t = part[0][lane];
#pragma unroll
    for (int k = 1; k < GRAM_RC; ++k) t += part[k][lane];
    W[i + (int64_t)j * ldw] = t;
    W[j + (int64_t)i * ldw] = t;
  }
}

template <int MAXS>
cudaError_t launch_diag(const double* A, int64_t lda, int64_t m, int n, const GramGeom& g, double* partial,
                        Lane s) {
  const size_t sm = (size_t)2 * KC * (n | 1) * sizeof(double);
  cudaError_t e = cudaFuncSetAttribute(k_gram_diag<MAXS>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)(2 * KC * 129 * sizeof(double)));
  if (e != cudaSuccess) return e;
  e = launch_chained(k_gram_diag<MAXS>, dim3((unsigned)g.nsplit), dim3(NT), sm, s, dim3(1),
                     chain_early(2 * g.nsplit), A, lda, m, n, g.rows_per_split, g.T, partial);
  if (e != cudaSuccess) return e;
  count_launch();
  return cudaGetLastError();
}

}  // namespace

namespace {
// CTAs of equal work per row range: one per off-diagonal tile, one per two
// diagonal tiles.
int64_t gram_items(int ntile) { return (int64_t)ntile * (ntile - 1) / 2 + ceil_div(ntile, 2); }
int gram_sms() {
  int dev = 0, sms = 148;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  return sms;
}
// CTAs resident on an SM at a time (few slots per thread).
int gram_resident(int n) {
  const int slots = gram_slots(std::min(n, 128));
  return slots <= 8 ? 3 : (slots <= 16 ? 2 : 1);
}
}  // namespace

GramGeom gram_geometry(int64_t m, int n, int64_t max_splits, int ctas_per_sm, int row_unit, bool shared) {
  GramGeom g;
  g.ntile = (int)ceil_div(n, 128);
  g.T = (int)ceil_div(ceil_div(n, g.ntile), 16) * 16;
  g.ntiles_total = g.ntile + g.ntile * (g.ntile - 1) / 2;
  const int sms = gram_sms();
  const int64_t items = gram_items(g.ntile);
  // CTAs per SM: one, and where several are resident at a time and each still
  // has 35000 clocks (17 us) of FP64 work, that many. More only cost: filling a
  // CTA's pipeline, writing its partial tiles and reading them back take 2 to
  // 3 us. Gram and sum together with 1, 2, 3, 4 CTAs per SM: 4096 x 64 29, 32, 41,
  // 41 us; 50021 x 100 435, 451, 463, 474 us; 131072 x 32 166, 145, 136, 171 us;
  // 262144 x 16 105, 93, 89, 125 us.
  const int resident = gram_resident(n), knob = std::max(1, ctas_per_sm);
  const double clocks = (double)m * n * (n + 1) / 2 / (2.0 * sms);
  const int64_t per_sm = std::min(knob, clocks >= 35000.0 * resident ? resident : 1);
  // as many ranges as fit in that many whole waves, none shorter than 8 rows;
  // on a shared lane more and shorter ones, none shorter than 32 rows
  int64_t want = std::min<int64_t>(per_sm * sms / items, m / 8);
  if (shared) want = std::min<int64_t>((int64_t)std::min(knob, GRAM_SHARED_WAVES) * sms / items, m / 32);
  want = std::max<int64_t>(1, want);
  if (max_splits > 0) want = std::min<int64_t>(want, max_splits);
  g.rows_per_split = ceil_div(ceil_div(m, want), row_unit) * row_unit;
  g.nsplit = std::max<int64_t>(1, ceil_div(m, g.rows_per_split));
  return g;
}

int64_t gram_split_capacity(int n, bool shared) {
  const int per_sm = shared ? GRAM_SHARED_WAVES : gram_resident(n);
  return std::max<int64_t>(1, (int64_t)per_sm * gram_sms() / gram_items((int)ceil_div(n, 128)));
}

cudaError_t gram_partials(const double* A, int64_t lda, int64_t m, int n, const GramGeom& g, double* partial,
                          Lane s) {
  if (g.ntile == 1) {
    const int slots = gram_slots(n);
    if (slots <= 8) return launch_diag<8>(A, lda, m, n, g, partial, s);
    if (slots <= 16) return launch_diag<16>(A, lda, m, n, g, partial, s);
    if (slots <= 24) return launch_diag<24>(A, lda, m, n, g, partial, s);
    return launch_diag<gram_slots(128)>(A, lda, m, n, g, partial, s);
  }
  constexpr size_t sm = (size_t)4 * KC * 129 * sizeof(double);
  cudaError_t e = cudaFuncSetAttribute(k_gram_tiles, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  if (e != cudaSuccess) return e;
  const int noff = g.ntiles_total - g.ntile;
  dim3 grid((unsigned)g.nsplit, (unsigned)(noff + ceil_div(g.ntile, 2)));
  k_gram_tiles<<<grid, NT, sm, s>>>(A, lda, m, n, g.rows_per_split, g.T, g.ntile, g.ntiles_total, partial);
  count_launch();
  return cudaGetLastError();
}

cudaError_t gram_reduce(const double* partial, const GramGeom& g, int n, double* W, int64_t ldw, Lane s) {
  dim3 block(32 * GRAM_RC);
  dim3 grid((unsigned)ceil_div(n, 32), (unsigned)n);
  cudaError_t e = launch_chained(k_gram_reduce, grid, block, 0, s, dim3(1), true, partial, g.nsplit, g.T, g.ntile,
                                 g.ntiles_total, n, W, ldw);
  if (e != cudaSuccess) return e;
  count_launch();
  return cudaGetLastError();
}

}  // namespace cqr2

namespace {

// Device address of g_noalloc_scratch, looked up once per CUDA context (with
// that context current) on the first call there, and cached. Host code must
// not use the symbol itself: on the host it names a stand-in, not device
// memory. The cache is keyed by the context's process-unique id
// (cuCtxGetId), so a context made current by the driver API, or the new
// primary context after a cudaDeviceReset, gets its own lookup instead of a
// stale address; where the driver lacks cuCtxGetId the key is the device
// ordinal (primary contexts only, no cudaDeviceReset in between).
typedef int (*CtxGetCurrentFn)(void**);
typedef int (*CtxGetIdFn)(void*, unsigned long long*);
constexpr int MAX_CONTEXTS = 64;
std::mutex g_scratch_mu;
struct ScratchEntry {
  unsigned long long key;
  double* addr;
};
ScratchEntry g_scratch[MAX_CONTEXTS];
int g_scratch_used = 0;

template <typename F>
F driver_fn(const char* name) {
  void* p = nullptr;
  cudaDriverEntryPointQueryResult q;
  if (cudaGetDriverEntryPoint(name, &p, cudaEnableDefault, &q) != cudaSuccess || q != cudaDriverEntryPointSuccess)
    return nullptr;
  return reinterpret_cast<F>(p);
}

// Key of the current context: its unique id with the top bit set, or the
// device ordinal when the driver cannot tell contexts apart (or no context is
// current yet; the entry point's pointer checks have made the runtime's
// context current by then).
cudaError_t context_key(unsigned long long* key) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  static CtxGetCurrentFn get_cur = driver_fn<CtxGetCurrentFn>("cuCtxGetCurrent");
  static CtxGetIdFn get_id = driver_fn<CtxGetIdFn>("cuCtxGetId");
  void* ctx = nullptr;
  unsigned long long id = 0;
  if (get_cur && get_id && get_cur(&ctx) == 0 && ctx && get_id(ctx, &id) == 0) {
    *key = id | (1ull << 63);
    return cudaSuccess;
  }
  *key = (unsigned long long)dev;
  return cudaSuccess;
}

cudaError_t noalloc_scratch(double** out) {
  unsigned long long key = 0;
  cudaError_t e = context_key(&key);
  if (e != cudaSuccess) return e;
  std::lock_guard<std::mutex> lk(g_scratch_mu);
  for (int i = 0; i < g_scratch_used; ++i)
    if (g_scratch[i].key == key) {
      *out = g_scratch[i].addr;
      return cudaSuccess;
    }
  if (g_scratch_used == MAX_CONTEXTS) return cudaErrorInvalidDevice;
  void* p = nullptr;
  e = cudaGetSymbolAddress(&p, cqr2::g_noalloc_scratch);
  if (e != cudaSuccess) return e;
  g_scratch[g_scratch_used++] = {key, static_cast<double*>(p)};
  *out = static_cast<double*>(p);
  return cudaSuccess;
}

// A pointer the kernels may dereference on the current device: device or
// managed memory of this device. Host and unregistered pointers, and memory
// of another device, are rejected (cudaPointerGetAttributes allocates
// nothing).
bool on_current_device(const void* ptr) {
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess) return false;
  cudaPointerAttributes a;
  if (cudaPointerGetAttributes(&a, ptr) != cudaSuccess) {
    cudaGetLastError();  // clear the error the failed query recorded
    return false;
  }
  return (a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged) && a.device == dev;
}

}  // namespace

extern "C" cqr2_status_t cqr2_syrk_noalloc(const double* dA, int64_t m, int64_t n, int64_t lda, double* dW,
                                           int64_t ldw, void* stream) {
  using namespace cqr2;
  if (!dA || !dW || n < 1 || m < n || lda < m || ldw < n) return CQR2_ERR_INVALID_ARG;
  if (n > CQR2_NOALLOC_MAX_N) return CQR2_ERR_UNSUPPORTED;
  if (!on_current_device(dA) || !on_current_device(dW)) return CQR2_ERR_INVALID_ARG;
  const GramGeom g0 = gram_geometry(m, (int)n, 0);
  const int64_t per_split = (int64_t)g0.ntiles_total * g0.T * g0.T;
  const int64_t max_splits = (int64_t)NOALLOC_DOUBLES / per_split;
  if (max_splits < 1) return CQR2_ERR_UNSUPPORTED;
  const GramGeom g = gram_geometry(m, (int)n, max_splits);
  if (g.partial_doubles() > NOALLOC_DOUBLES) return CQR2_ERR_UNSUPPORTED;
  double* scratch = nullptr;
  if (noalloc_scratch(&scratch) != cudaSuccess) return CQR2_ERR_CUDA;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  // Every partial entry the reduction reads is written by gram_partials in
  // this same call, so nothing left over from an earlier call is used and no
  // clearing is needed.
  if (gram_partials(dA, lda, m, (int)n, g, scratch, s) != cudaSuccess) return CQR2_ERR_CUDA;
  if (gram_reduce(scratch, g, (int)n, dW, ldw, s) != cudaSuccess) return CQR2_ERR_CUDA;
  return CQR2_OK;
}
