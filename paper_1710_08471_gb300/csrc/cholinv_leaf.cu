// CholInv of a leaf, n <= CHOLINV_LEAF = 128 (Algorithm 1's recursion stops
// here): W = L L^T, Y = L^-1, in one launch of one thread-block cluster.
//
// What decides the design is how FP64 issues on GB300: an FP64 instruction
// occupies its SM partition's pipe for 64 clocks and has 64 clocks of latency,
// so the n pivots are a chain of FP64 latencies, and the 2 n^3 / 3 flops of
// the trailing updates need several SMs to stay behind it (at n = 128 one SM
// would take 175 us for them).
//
// Blocked by 8, right-looking, in the form W = Lu D Lu^T with unit lower Lu,
// whose pivot chain needs a reciprocal and one product where the square-root
// form needs a reciprocal square root and two scalings:
//   step p:  V(i) = A(i,p) Lu_pp^-T,  Lu(i) = V(i) D_p^-1
//            A(i,j) -= Lu(i) V(j)^T          for p < j <= i
//            Tu(p,j) = Lu_pp^-1 Tu(p,j)      for j < p: a finished row of Lu^-1
//            Tu(i,j) -= Lu(i) Tu(p,j)        for j <= p < i, with Tu(p,p) = Lu_pp^-1
// (both solves by substitution) and L = Lu D^(1/2), Y = D^(-1/2) Lu^-1. A(i,j)
// is live until step j and Tu(i,j) from step j on, so one 8 x 8 tile of shared
// memory holds both.
//
// Block columns are dealt to the cluster's CTAs in a snake (0..C-1, C-1..0),
// which evens out their work. At step p the owner of block column p+1 first
// brings that column up to date; one warp factors its diagonal tile while six
// others follow it column by column with V and Lu of the tiles below, and send
// Lu to every CTA of the cluster and V(j) to the owner of column j (distributed
// shared memory). Only then does it join the others in the rest of step p. One
// split cluster barrier per step: a CTA arrives when it has entered the step
// (the owner, when its panel is sent) and waits when it has finished it, so
// panels live in three slots (a panel is overwritten two steps after every CTA
// has arrived past its last use).
//
// Measured, us per CholInv back to back (before: one CTA per 64 columns with a
// rank-1 step and a block barrier per column, GEMM launches above that):
// n = 16: 22 -> 13, 32: 37 -> 21, 64: 64 -> 39, 100: 222 -> 72, 128: 238 -> 99.
#include <algorithm>
#include <type_traits>

#include "fp64_rsqrt.cuh"
#include "kernels.h"

namespace cqr2 {
namespace {

constexpr int TB = 8;             // block size
constexpr int TLD = 10;           // row pitch of a tile: 16-byte loads of 8 rows hit distinct banks
constexpr int TSZ = TB * TLD;     // doubles per tile
constexpr int LT = 256, LW = LT / 32;
constexpr int SLOTS = 3;
constexpr int MAXC = 8;           // portable cluster size
constexpr int MAXB = CHOLINV_LEAF / TB;

__device__ __forceinline__ uint32_t s_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ uint32_t cluster_size() {
  uint32_t r;
  asm("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
// Stores to the same shared-memory offset in CTA `rank` of the cluster.
__device__ __forceinline__ uint32_t remote(uint32_t addr, uint32_t rank) {
  uint32_t a;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(addr), "r"(rank));
  return a;
}
__device__ __forceinline__ void st_remote(uint32_t addr, uint32_t rank, double v) {
  asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(remote(addr, rank)), "d"(v) : "memory");
}
__device__ __forceinline__ void st_remote(uint32_t addr, uint32_t rank, double2 v) {
  asm volatile("st.shared::cluster.v2.f64 [%0], {%1, %2};" ::"r"(remote(addr, rank)), "d"(v.x), "d"(v.y) : "memory");
}

// Lane (r, g), r = lane & 7, g = lane >> 3, holds elements (r, 2g) and (r, 2g + 1) of a tile.
typedef double2 Pair;
__device__ __forceinline__ Pair tile_get(const double* t, int r, int g) {
  return *reinterpret_cast<const double2*>(t + r * TLD + 2 * g);
}
__device__ __forceinline__ void tile_put(double* t, int r, int g, Pair v) {
  *reinterpret_cast<double2*>(t + r * TLD + 2 * g) = v;
}

// acc(r, c) -= sum over k in [K0, K0 + KN) of A(r, k) B(c, k)
template <int K0 = 0, int KN = TB>
__device__ __forceinline__ void tile_sub(Pair& acc, const double* A, const double* B, int r, int g) {
  double2 x[KN / 2], y[KN / 2], z[KN / 2];
#pragma unroll
  for (int q = 0; q < KN / 2; ++q) {
    x[q] = *reinterpret_cast<const double2*>(A + r * TLD + K0 + 2 * q);
    y[q] = *reinterpret_cast<const double2*>(B + 2 * g * TLD + K0 + 2 * q);
    z[q] = *reinterpret_cast<const double2*>(B + (2 * g + 1) * TLD + K0 + 2 * q);
  }
#pragma unroll
  for (int q = 0; q < KN / 2; ++q) {
    acc.x = fma(-x[q].x, y[q].x, acc.x);
    acc.y = fma(-x[q].x, z[q].x, acc.y);
    acc.x = fma(-x[q].y, y[q].y, acc.x);
    acc.y = fma(-x[q].y, z[q].y, acc.y);
  }
}

struct LeafSmem {
  double* tiles;  // own block columns, tile (i, j) at base(j) + (i - j) TSZ
  double* V;      // [SLOTS][blocks][TSZ]: V(j) of own columns
  double* Lu;     // [SLOTS][blocks][TSZ]: Lu(i), the diagonal tile included
  double* Z;      // [2][TSZ]: inverse of Lu's diagonal tile of own columns (one CTA may own p and p + 1)
  double* half;   // [TSZ]: half of a diagonal tile's update
  double* Tr;     // [own columns][TSZ]: Tu(p, j) as [column][k]
  double* dg;     // [SLOTS][2 TB]: D; the owner also keeps 1/D
};

// Named barriers: 1 joins the two halves of a diagonal tile's update; PANEL_BAR
// + k (k < TB) tells the panel warps that column k of the factored diagonal
// tile is there, PANEL_BAR + TB that the tile has been factored again with
// divisions. Warp 0 factors and PW = 6 warps solve panel tiles; warp 4, on
// warp 0's SM partition, stays out. (With three panel warps the factorization
// runs undisturbed, 4000 clocks against up to 5000, but the panel then takes
// longer than it: 45 against 41 us at n = 64, 126 against 102 us at n = 128,
// with 21 FP64 instructions to a panel tile; it has 15 now.)
constexpr int PW = 6, PANEL_BAR = 2, PANEL_THREADS = 32 * (1 + PW);
__device__ __forceinline__ void bar_arrive(int id) {
  asm volatile("bar.arrive %0, %1;" ::"r"(id), "n"(PANEL_THREADS) : "memory");
}
__device__ __forceinline__ void bar_wait(int id) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "n"(PANEL_THREADS) : "memory");
}

// The diagonal tile's factorization with divisions, for pivots outside the
// reciprocal's range and for breakdowns (reported, and spread as NaN).
__device__ __noinline__ void factor_tile_div(double* t, Pair e, double* Ld, double* Z, double* dd, int lane, int nlive,
                                             DevStatus* st, int pass, long long off) {
  const int r = lane & 7, g = lane >> 3, c0 = 2 * g, c1 = 2 * g + 1;
  __syncwarp();
  tile_put(t, r, g, e);
  Pair l{0.0, 0.0};
  __syncwarp();
#pragma unroll 1
  for (int k = 0; k < TB; ++k) {
    double d = t[k * TLD + k];
    const double ar = t[r * TLD + k];
    const double b0 = t[max(c0, k) * TLD + min(c0, k)], b1 = t[max(c1, k) * TLD + min(c1, k)];
    if (!(d > 0.0) || !isfinite(d)) {
      if (lane == 0 && k < nlive) report_pivot(st, pass, off + k, d);
      d = __longlong_as_double(0x7FF8000000000000ll);
    }
    if (lane == 0) dd[k] = d;
    const double w = ar / d;
    if (c0 == k) l.x = w;
    if (c1 == k) l.y = w;
    __syncwarp();
    if (r > k) {
      e.x = fma(-w, c0 == k ? 1.0 : b0, c0 == k ? 0.0 : e.x);
      e.y = fma(-w, c1 == k ? 1.0 : b1, c1 == k ? 0.0 : e.y);
      tile_put(t, r, g, e);
    }
    __syncwarp();
  }
  tile_put(Z, r, g, {c0 < r ? e.x : (c0 == r ? 1.0 : 0.0), c1 < r ? e.y : (c1 == r ? 1.0 : 0.0)});
  tile_put(Ld, r, g, {c0 < r ? l.x : (c0 == r ? 1.0 : 0.0), c1 < r ? l.y : (c1 == r ? 1.0 : 0.0)});
}

// Factors the diagonal tile (this lane's elements e, t its shared memory): Z,
// Lu and D of the block (dd: D, then its reciprocals). Warp 0. Each lane forms
// the pivot's reciprocal itself. A step's chain is one FMA (the element of
// column k + 1 first), its exchange through shared memory, the reciprocal in
// integers and the product; the other element's FMA runs beside the next
// reciprocal, and nothing on the chain branches: the pivots' range is looked at
// once, at the end. Lu's columns are published step by step for the panel warps.
__device__ __forceinline__ void factor_tile(double* t, Pair e, double* Ld, double* Z, double* dd, int* exact, int lane,
                                            int nlive, DevStatus* st, int pass, long long off) {
  const int r = lane & 7, g = lane >> 3, c0 = 2 * g, c1 = 2 * g + 1;
  const Pair e0 = e;
  bool ok = true;
  tile_put(t, r, g, e);
  tile_put(Ld, r, g, {c0 == r ? 1.0 : 0.0, c1 == r ? 1.0 : 0.0});
  __syncwarp();
  double d = t[0];
#pragma unroll
  for (int k = 0; k < TB; ++k) {
    const double y = pivot_rcp(d);
    ok = ok && pivot_rcp_ok(d);
    __syncwarp();  // step k - 1's elements are all in place
    const double ar = t[r * TLD + k];
    const double b0 = t[(c0 > k ? c0 : k) * TLD + (c0 > k ? k : c0)];
    const double b1 = t[(c1 > k ? c1 : k) * TLD + (c1 > k ? k : c1)];
    const double w = ar * y;  // Lu's column k
    const bool below = r > k;
    const double s0 = c0 == k ? 1.0 : b0, s1 = c1 == k ? 1.0 : b1;
    const double f0 = c0 == k ? 0.0 : e.x, f1 = c1 == k ? 0.0 : e.y;
    const double nw = below ? -w : 0.0;
    auto first = [&] {
      const double v = fma(nw, s0, f0);
      if (below) t[r * TLD + c0] = e.x = v;
    };
    auto second = [&] {
      const double v = fma(nw, s1, f1);
      if (below) t[r * TLD + c1] = e.y = v;
    };
    __syncwarp();  // the step's reads are done
    if (k < TB - 1) {
      if ((k + 1) & 1) second();
      else first();
      __syncwarp();
    }
    const double dk = d;
    if (k < TB - 1) {
      d = t[(k + 1) * TLD + k + 1];
      if ((k + 1) & 1) first();
      else second();
    }
    if (below && (c0 == k || c1 == k)) Ld[r * TLD + k] = w;
    if (lane == 0) {
      dd[k] = dk;
      dd[TB + k] = y;
      if (k == TB - 1) *exact = !ok;
    }
    __syncwarp();
    bar_arrive(PANEL_BAR + k);
  }
  if (!ok) {
    factor_tile_div(t, e0, Ld, Z, dd, lane, nlive, st, pass, off);
    __syncwarp();
    bar_wait(PANEL_BAR + TB);
    return;
  }
  tile_put(Z, r, g, {c0 < r ? e.x : (c0 == r ? 1.0 : 0.0), c1 < r ? e.y : (c1 == r ? 1.0 : 0.0)});  // unit lower
}

__global__ void __launch_bounds__(LT, 1)
    k_cholinv_leaf(const double* W, int64_t ldw, int n, double* L, int64_t ldl, double* Y, int64_t ldy, double* Rt,
                   int64_t ldrt, double* Rp, int rpw, DevStatus* st, int pass, long long off) {
  grid_chain();
  extern __shared__ __align__(16) double smem[];
  __shared__ int s_exact;  // a pivot of the panel factored last needs real divisions
  const int C = (int)cluster_size(), me = (int)cluster_rank();
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31, r = lane & 7, g = lane >> 3;
  const int nb = (n + TB - 1) / TB, rpp = rpw + (rpw & 1);
  const int rpl = rpw > 0 ? (n + rpw - 1) / rpw * rpw - n : 0;  // R^-1's packing: pitch rpp, the first group lacks rpl columns
  // own block columns: q-th is q C + (q even ? me : C - 1 - me)
  auto column = [&](int q) { return q * C + ((q & 1) ? C - 1 - me : me); };
  auto owner = [&](int j) {
    const int x = j % C;
    return ((j / C) & 1) ? C - 1 - x : x;
  };
  LeafSmem sm;
  sm.V = smem;
  sm.Lu = sm.V + SLOTS * nb * TSZ;
  sm.Z = sm.Lu + SLOTS * nb * TSZ;
  sm.half = sm.Z + 2 * TSZ;
  sm.dg = sm.half + TSZ;
  sm.Tr = sm.dg + SLOTS * 2 * TB;
  sm.tiles = sm.Tr + ((nb + C - 1) / C) * TSZ;
  auto tile_base = [&](int q) {  // tiles of own columns before the q-th
    int b = 0;
    for (int u = 0; u < q; ++u) b += nb - column(u);
    return sm.tiles + b * TSZ;
  };
  auto slot_tile = [&](double* base, int p, int i) { return base + ((p % SLOTS) * nb + i) * TSZ; };

  // ---- load the own columns (lower triangle; identity beyond n)
  for (int q = 0; column(q) < nb; ++q) {
    const int j = column(q), rows = (nb - j) * TB;
    double* tb = tile_base(q);
    for (int e = t; e < rows * TB; e += LT) {
      const int i = e % rows, c = e / rows;  // row j TB + i, column j TB + c
      const int gi = j * TB + i, gj = j * TB + c;
      double v = 0.0;
      if (gi < n && gj <= gi) v = W[gi + (int64_t)gj * ldw];
      if (gi >= n && gi == gj) v = 1.0;
      tb[(i / TB) * TSZ + (i % TB) * TLD + c] = v;
    }
  }
  __syncthreads();
  // W has been read everywhere (it may share storage with an output) and
  // every CTA of the cluster runs (its shared memory may be written)
  cluster_arrive();
  cluster_wait();

  // Block column p (its tiles tb): the last update (from panel p - 1, unless p
  // is 0), the diagonal tile's factorization, V and Lu of the tiles below it,
  // and their way to the cluster. Run by the owner's whole CTA.
  auto lead_column = [&](int p) {
    double* tb = tile_base(p / C);
    double* Ld = slot_tile(sm.Lu, p, p);
    double* dd = sm.dg + (p % SLOTS) * 2 * TB;
    double* Z = sm.Z + (p & 1) * TSZ;
    const double* Vn = p ? slot_tile(sm.V, p - 1, p) : nullptr;
    const uint32_t at = (uint32_t)((r * TLD + 2 * g) * sizeof(double));
    if (warp == 0) {
      Pair e = tile_get(tb, r, g);
      if (p) {  // on the chain: warp 1 takes half of the products
        Pair h{0.0, 0.0};
        tile_sub<0, TB / 2>(h, slot_tile(sm.Lu, p - 1, p), Vn, r, g);
        asm volatile("bar.sync 1, 64;" ::: "memory");
        const Pair h1 = tile_get(sm.half, r, g);
        e.x += h.x + h1.x;
        e.y += h.y + h1.y;
      }
      factor_tile(tb, e, Ld, Z, dd, &s_exact, lane, n - p * TB, st, pass, off + (long long)p * TB);
      __syncwarp();
      const Pair ld = tile_get(Ld, r, g);
      const double dl = dd[lane & (TB - 1)];
      for (int c = 0; c < C; ++c)
        if (c != me) {
          st_remote(s_addr(Ld) + at, c, ld);
          if (lane < TB) st_remote(s_addr(dd + lane), c, dl);
        }
    } else if (warp != 4) {
      if (p && warp == 1) {
        Pair h{0.0, 0.0};
        tile_sub<TB / 2, TB / 2>(h, slot_tile(sm.Lu, p - 1, p), Vn, r, g);
        tile_put(sm.half, r, g, h);
        asm volatile("bar.sync 1, 64;" ::: "memory");
      }
      constexpr int MAXU = (MAXB - 1 + PW - 1) / PW;
      const int pw = warp == 1 ? PW - 1 : (warp < 4 ? warp - 2 : warp - 3);  // warp 1 has half the diagonal's update too
      const int i0 = p + 1 + pw, nt = i0 < nb ? (nb - 1 - i0) / PW + 1 : 0;
      Pair v[MAXU], l[MAXU];
      auto solve = [&](auto tiles) {
        constexpr int U = decltype(tiles)::value;
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const int i = i0 + u * PW;
          double* tl = tb + (i - p) * TSZ;
          v[u] = tile_get(tl, r, g);
          if (p) tile_sub(v[u], slot_tile(sm.Lu, p - 1, i), Vn, r, g);
          tile_put(tl, r, g, v[u]);  // for a second solve with divisions
        }
        // V(r, c) -= V(r, k) Lu(c, k): column k is final once the columns before it are subtracted
#pragma unroll
        for (int k = 0; k < TB; ++k) {
          bar_wait(PANEL_BAR + k);
          if (k == TB - 1) break;
          const double b0 = Ld[2 * g * TLD + k], b1 = Ld[(2 * g + 1) * TLD + k];
#pragma unroll
          for (int u = 0; u < U; ++u) {
            const double vk = __shfl_sync(0xffffffffu, (k & 1) ? v[u].y : v[u].x, r + 8 * (k >> 1));
            if (k < 6) v[u].x = 2 * g > k ? fma(-vk, b0, v[u].x) : v[u].x;
            v[u].y = 2 * g + 1 > k ? fma(-vk, b1, v[u].y) : v[u].y;
          }
        }
        const Pair y = *reinterpret_cast<const double2*>(dd + TB + 2 * g);
#pragma unroll
        for (int u = 0; u < U; ++u) l[u] = {v[u].x * y.x, v[u].y * y.y};
      };
      if (nt == 0) {
        for (int k = 0; k < TB; ++k) bar_wait(PANEL_BAR + k);
      } else if (nt == 1) {
        solve(std::integral_constant<int, 1>());
      } else if (nt == 2) {
        solve(std::integral_constant<int, 2>());
      } else {
        solve(std::integral_constant<int, MAXU>());
      }
      static_assert(MAXU == 3, "cases above");
      const bool again = s_exact != 0;
      if (again) bar_wait(PANEL_BAR + TB);
#pragma unroll
      for (int u = 0; u < MAXU; ++u) {
        if (u >= nt) break;
        const int i = i0 + u * PW;
        if (again) {
          v[u] = tile_get(tb + (i - p) * TSZ, r, g);
#pragma unroll
          for (int k = 0; k < TB - 1; ++k) {
            const double vk = __shfl_sync(0xffffffffu, (k & 1) ? v[u].y : v[u].x, r + 8 * (k >> 1));
            if (2 * g > k) v[u].x = fma(-vk, Ld[2 * g * TLD + k], v[u].x);
            if (2 * g + 1 > k) v[u].y = fma(-vk, Ld[(2 * g + 1) * TLD + k], v[u].y);
          }
          l[u] = {v[u].x / dd[2 * g], v[u].y / dd[2 * g + 1]};
        }
        double* Vi = slot_tile(sm.V, p, i);
        double* Li = slot_tile(sm.Lu, p, i);
        const int o = owner(i);
        tile_put(Li, r, g, l[u]);
        if (o == me) tile_put(Vi, r, g, v[u]);
        else st_remote(s_addr(Vi) + at, o, v[u]);
        for (int c = 0; c < C; ++c)
          if (c != me) st_remote(s_addr(Li) + at, c, l[u]);
      }
    }
    __syncwarp();
  };

  // zeros above L's and Y's diagonal tiles, below R's, and in R^-1's packing:
  // by the CTAs (with one CTA: the warps) that do not start the chain
  {
    const int who = C > 1 ? (me - 1) * LT + t : t - 32, stride = C > 1 ? (C - 1) * LT : LT - 32;
    if (who >= 0) {
      for (int e = who; e < n * n; e += stride) {
        const int i = e % n, j = e / n;
        if (i < j) {
          L[i + (int64_t)j * ldl] = 0.0;
          Y[i + (int64_t)j * ldy] = 0.0;
        }
        if (i > j && Rt != nullptr) Rt[i + (int64_t)j * ldrt] = 0.0;
      }
      if (Rp != nullptr)
        for (int e = who; e < RP_GROUPS * n * rpp; e += stride) {
          const int c = e % rpp, k = (e / rpp) % n, col = (e / (rpp * n)) * rpw + c - rpl;
          if (c >= rpw || col < 0 || col >= n || k > col) Rp[e] = 0.0;
        }
    }
  }
  if (owner(0) == me) lead_column(0);
  cluster_arrive();
  cluster_wait();

  for (int p = 0; p < nb; ++p) {
    __syncthreads();  // the CTA's work of step p - 1 is complete
    const int nx = p + 1;
    const bool lead = nx < nb && owner(nx) == me;
    const int qn = lead ? nx / C : -1;  // index of column nx among the own ones
    if (lead) lead_column(nx);
    cluster_arrive();
    // ---- the rest of step p
    const double* D = sm.dg + (p % SLOTS) * 2 * TB;
    const double* Ld = slot_tile(sm.Lu, p, p);
    int turn = 0;  // tasks are dealt to the warps in turn
    // finished row p of Lu^-1: the updates' right operand, and Y's row
    for (int q = 0; column(q) <= p && column(q) < nb; ++q) {
      if ((turn++ & (LW - 1)) != warp) continue;
      const int j = column(q);
      double* Tj = sm.Tr + q * TSZ;
      Pair v;
      if (j == p) {
        v = tile_get(sm.Z + (p & 1) * TSZ, r, g);
      } else {
        v = tile_get(tile_base(q) + (p - j) * TSZ, r, g);
#pragma unroll
        for (int k = 0; k < TB - 1; ++k) {
          const double t0 = __shfl_sync(0xffffffffu, v.x, k + 8 * g), t1 = __shfl_sync(0xffffffffu, v.y, k + 8 * g);
          const double w = Ld[r * TLD + k];
          if (r > k) {
            v.x = fma(-w, t0, v.x);
            v.y = fma(-w, t1, v.y);
          }
        }
      }
      Tj[2 * g * TLD + r] = v.x;
      Tj[(2 * g + 1) * TLD + r] = v.y;
      double s, unused;
      chol_rsqrt_tight(D[r], &s, &unused);
      const int gi = p * TB + r;
      if (gi < n) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int gj = j * TB + 2 * g + h;
          if (gj > gi) continue;
          const double y = (h ? v.y : v.x) * s;
          Y[gi + (int64_t)gj * ldy] = y;
          if (Rp != nullptr) Rp[((int64_t)((gi + rpl) / rpw) * n + gj) * rpp + (gi + rpl) % rpw] = y;  // R^-1(gj, gi)
        }
      }
    }
    // Column p of L and row p of R, as Lu D^(1/2) and not V D^(-1/2): Y comes
    // from the same rounded Lu, so L Y = I holds to the last roundings, which
    // is what R2 R1 needs of it.
    if (owner(p) == me) {
      double s0 = 0.0, s1 = 0.0;
      for (int i = p; i < nb; ++i) {
        if ((turn++ & (LW - 1)) != warp) continue;
        if (s0 == 0.0) {
          double unused;
          chol_rsqrt_tight(D[2 * g], &unused, &s0);
          chol_rsqrt_tight(D[2 * g + 1], &unused, &s1);
        }
        const Pair v = tile_get(slot_tile(sm.Lu, p, i), r, g);
        const int gi = i * TB + r;
        if (gi >= n) continue;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int gj = p * TB + 2 * g + h;
          if (gj > gi) continue;
          const double l = h ? v.y * s1 : v.x * s0;
          L[gi + (int64_t)gj * ldl] = l;
          if (Rt != nullptr) Rt[gj + (int64_t)gi * ldrt] = l;
        }
      }
    }
    __syncthreads();
    for (int q = 0; column(q) < nb; ++q) {
      const int j = column(q);
      if (q == qn) continue;  // brought up to date above
      double* tb = tile_base(q);
      const double* B = j > p ? slot_tile(sm.V, p, j) : sm.Tr + q * TSZ;
      for (int i = j > p ? j : nx; i < nb; ++i) {
        if ((turn++ & (LW - 1)) != warp) continue;
        double* tl = tb + (i - j) * TSZ;
        // a diagonal tile's entries are far larger than the products: those are
        // summed first, one rounding at the entries' magnitude instead of eight
        const bool apart = i == j;
        const Pair e = tile_get(tl, r, g);
        Pair h = apart || j == p ? Pair{0.0, 0.0} : e;
        tile_sub(h, slot_tile(sm.Lu, p, i), B, r, g);
        if (apart) {
          h.x += e.x;
          h.y += e.y;
        }
        tile_put(tl, r, g, h);
      }
    }
    cluster_wait();
  }
}

size_t leaf_smem(int n, int C) {
  const int nb = (n + TB - 1) / TB;
  // the CTA with the most tiles
  int most = 0;
  for (int me = 0; me < C; ++me) {
    int tiles = 0;
    for (int q = 0;; ++q) {
      const int j = q * C + ((q & 1) ? C - 1 - me : me);
      if (j >= nb) break;
      tiles += nb - j;
    }
    most = std::max(most, tiles);
  }
  return ((size_t)(2 * SLOTS * nb + 3 + (nb + C - 1) / C + most) * TSZ + SLOTS * 2 * TB) * sizeof(double);
}

constexpr int LEAF_SMEM_MAX = 96 * 1024;

}  // namespace

// CTAs of the cluster: as many as there are block columns, in powers of two up
// to the portable 8. Measured (us per CholInv back to back, launch included):
// n = 16: 15.0 with 1 CTA, 12.7 with 2; n = 32: 23.8 with 2, 20.4 with 4;
// n = 64: 90 with 1, 53 with 2, 41 with 4, 38 with 8; n = 128: 121 with 4, 102 with 8.
static int leaf_ctas(int n) {
  int c = 1;
  while (c < MAXC && 2 * c <= (n + TB - 1) / TB) c *= 2;
  return c;
}

cudaError_t cholinv_leaf(int n, const double* W, int64_t ldw, double* L, int64_t ldl, double* Y, int64_t ldy,
                         double* Rt, int64_t ldrt, double* Rp, int rpw, DevStatus* st, int pass, long long off,
                         Lane s) {
  if (n < 1 || n > CHOLINV_LEAF) return cudaErrorInvalidValue;
  const int C = leaf_ctas(n);
  const size_t sm = leaf_smem(n, C);
  if (sm > LEAF_SMEM_MAX) return cudaErrorInvalidValue;
  cudaError_t e = cudaFuncSetAttribute(k_cholinv_leaf, cudaFuncAttributeMaxDynamicSharedMemorySize, LEAF_SMEM_MAX);
  if (e != cudaSuccess) return e;
  e = launch_chained(k_cholinv_leaf, dim3((unsigned)C), dim3(LT), sm, s, dim3((unsigned)C), true, W, ldw, n, L, ldl, Y,
                     ldy, Rt, ldrt, Rp, rpw, st, pass, off);
  if (e != cudaSuccess) return e;
  count_launch();
  return cudaGetLastError();
}

}  // namespace cqr2
