// Internal helpers shared by the CholeskyQR2 kernels (not part of the C ABI).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace cqr2 {

// Device-side outcome of a factorization, written by the CholInv base-case
// kernel on the first non-positive or non-finite pivot. `lock` makes the
// first reporter win; later breakdowns (which see NaNs) are ignored.
struct DevStatus {
  int status;  // 0 = ok, 2 = not SPD
  int pass;    // CholeskyQR pass (1 or 2)
  long long pivot;
  double value;
  int lock;
  int pad;
};

__device__ __forceinline__ void report_pivot(DevStatus* st, int pass, long long pivot, double v) {
  if (atomicCAS(&st->lock, 0, 1) == 0) {
    st->status = 2;
    st->pass = pass;
    st->pivot = pivot;
    st->value = v;
  }
}

// 8-byte asynchronous global->shared copy; src_bytes = 0 zero-fills the
// destination without reading `src` (which must still be a valid address).
__device__ __forceinline__ void cp_async8(void* smem, const void* gmem, int src_bytes) {
  unsigned s = static_cast<unsigned>(__cvta_generic_to_shared(smem));
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;\n" ::"r"(s), "l"(gmem), "r"(src_bytes));
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;\n" ::"n"(N));
}

// The stream a call's kernels go to, and whether other calls' kernels run
// beside them (cqr2_plan_set_shared). Launch shapes are chosen for a call that
// has the GPU to itself; a shared lane takes what lets the streams interleave:
// no grid is set up early (it holds its slots while it waits), no product
// splits k over a cluster (which starts only where several SMs of a group have
// room at once), the Gram's ranges and the Q-form's panels go in shorter CTAs
// (between which the other streams' kernels start; a whole-wave Gram CTA holds
// its SM for up to 14 ms). Median latency of 500 FP64 least-squares requests at
// 100/s on 8 slots, three arrival seeds, ms: 15.8, 25.5, 44.8 with the shapes of
// a call alone and 14.0, 19.9, 40.7 shared; with early set-up 14.0, 22.1, 42.3,
// with k splits 14.2, 20.9, 41.3, with the Gram in one wave 14.3, 21.5, 40.7, with
// the Q-form in one wave 13.9, 20.4, 41.3. One request at a time then takes 0.7%
// longer.
struct Lane {
  cudaStream_t s;
  bool shared;
  Lane(cudaStream_t s_, bool shared_ = false) : s(s_), shared(shared_) {}
  operator cudaStream_t() const { return s; }
};

// The kernels of a factorization follow one another on one stream, and the
// small ones take a few microseconds each, about as long as the stream needs
// to drain one grid and start the next. They are launched with launch_chained,
// which lets a grid be set up on the SMs while its predecessor still runs, and
// open with grid_chain(): wait until the predecessor has completed and its
// writes are visible, then let the successor be set up. Since no grid ends
// before its own wait, completion stays in stream order, also for what is read
// and overwritten. The sources of these kernels hold no __ldg and no
// __restrict__: the read-only path is for data that stays constant during the
// kernel's lifetime, which begins before the wait, and such a load could be
// moved above it. (us per pass, whole factorizations: least squares of
// 1024 x 16 79 -> 61, 4096 x 64 202 -> 192, least squares of 131601 x 256 in
// split precision 2035 -> 2006.)
__device__ __forceinline__ void grid_chain() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// Whether a grid of that many CTAs, each of some tens of microseconds or more
// (Gram, Q-form, GEMM, Q^T b), is set up early. One that fills the SMs is not:
// while its predecessor holds some of them, its CTAs pile up on the rest.
// (777 columns in FP64: 15.4 ms, with every GEMM set up early 16.1. The Gram and
// the Q-form pass twice their CTAs: these run for long on an SM each, and at
// 4096 x 64 early ones cost 10 us. The 128 x 128 GEMMs of CholInv gain at up to
// an SM each, 12 us of 2017 at 131601 x 256.) Kernels whose CTAs last a
// microsecond or so (sums of partials, packing, transposition, copies,
// R2 R1) are set up early at any size: held to this rule too, 3000 x 80 took 235
// us instead of 231, 4096 x 128 503 instead of 499, 8192 x 200 1668 instead of
// 1657, and from 400 columns on nothing changed by more than 0.2%.
inline bool chain_early(int64_t ctas) {
  int dev = 0, sms = 152;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  return ctas <= sms;
}

// Launches kern (as a cluster where that has more than one CTA).
template <typename... P, typename... Args>
cudaError_t launch_chained(void (*kern)(P...), dim3 grid, dim3 block, size_t smem, Lane s, dim3 cluster, bool early,
                           Args... args) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at[2]{};
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = early && !s.shared ? 1 : 0;
  at[1].id = cudaLaunchAttributeClusterDimension;
  at[1].val.clusterDim.x = cluster.x;
  at[1].val.clusterDim.y = cluster.y;
  at[1].val.clusterDim.z = cluster.z;
  cfg.attrs = at;
  cfg.numAttrs = cluster.x * cluster.y * cluster.z > 1 ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, kern, static_cast<P>(args)...);
}

inline int64_t ceil_div(int64_t a, int64_t b) { return (a + b - 1) / b; }

}  // namespace cqr2
