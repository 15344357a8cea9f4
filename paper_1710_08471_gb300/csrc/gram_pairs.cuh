// The diagonal Gram tile's work list, shared by the Gram kernel and the fused
// Q-form + Gram kernel.
//
// A w x w diagonal tile has w (w + 1) / 2 entries on and above the diagonal.
// They are numbered row by row, and thread t of GRAM_NT owns entries t,
// t + GRAM_NT, .... FP64 issue is the bound and a warp instruction costs the
// same whatever its lane mask, so a warp runs exactly as many slots as hold
// one of its entries: whole groups of eight slots first, each with its own
// pass over the rows (the accumulators stay in registers, and a warp starts
// one FP64 instruction per 64 clocks anyway, so eight chains are plenty), and
// then a group of the one to seven that remain. Rounding w up to 32, 64 or 128
// instead, as a fixed set of three kernels did, made a 100-column Gram do 1.63
// times its work; a kernel per slot count took minutes to compile.
#pragma once

#include <stdint.h>

namespace cqr2 {

constexpr int GRAM_NT = 256;

__host__ __device__ constexpr int gram_slots(int w) { return (w * (w + 1) / 2 + GRAM_NT - 1) / GRAM_NT; }

// MAXS: the largest gram_slots(w) served.
template <int MAXS>
struct GramPairs {
  int oi[MAXS], oj[MAXS];
  double acc[MAXS];
  int cnt;    // this warp's slots
  int mine;   // this thread's entries
  __device__ __forceinline__ void init(int t, int w) {
    const int P = w * (w + 1) / 2;
    cnt = max(0, (P - (t & ~31) + GRAM_NT - 1) / GRAM_NT);
    mine = max(0, (P - t + GRAM_NT - 1) / GRAM_NT);
    int i = 0, start = 0;  // start: number of row i's first entry
#pragma unroll
    for (int s = 0; s < MAXS; ++s) {
      const int p = min(t + s * GRAM_NT, P - 1);
      while (p >= start + (w - i)) {
        start += w - i;
        ++i;
      }
      oi[s] = i;
      oj[s] = i + (p - start);
      acc[s] = 0.0;
    }
  }
  // slots G .. G + N - 1 over `rows` rows (a multiple of 4) at `pitch` doubles
  template <int G, int N>
  __device__ __forceinline__ void pass(const double* X, int pitch, int rows) {
    for (int k = 0; k < rows; k += 4)
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const double* x = X + (k + u) * pitch;
#pragma unroll
        for (int s = G; s < G + N; ++s) acc[s] = fma(x[oi[s]], x[oj[s]], acc[s]);
      }
  }
  template <int G, int N>
  __device__ __forceinline__ void rest(const double* X, int pitch, int rows) {
    if constexpr (N > 0) {
      if (cnt - G == N) pass<G, N>(X, pitch, rows);
      else rest<G, N - 1>(X, pitch, rows);
    }
  }
  template <int G>
  __device__ __forceinline__ void groups(const double* X, int pitch, int rows) {
    if constexpr (G + 8 <= MAXS) {
      if (cnt >= G + 8) {
        pass<G, 8>(X, pitch, rows);
        groups<G + 8>(X, pitch, rows);
      } else {
        rest<G, 7>(X, pitch, rows);
      }
    } else if constexpr (G < MAXS) {
      rest<G, MAXS - G>(X, pitch, rows);
    }
  }
  __device__ __forceinline__ void add(const double* X, int pitch, int rows) { groups<0>(X, pitch, rows); }
  // the tile's entries, column-major with leading dimension ld
  __device__ __forceinline__ void store(double* out, int ld) const {
#pragma unroll
    for (int s = 0; s < MAXS; ++s)
      if (s < mine) out[oi[s] + oj[s] * ld] = acc[s];
  }
};

}  // namespace cqr2
