// Deterministic block and grid reductions (fixed summation order for a fixed
// grid: per-block partials, then the last block to finish sums the partials
// in index order).
#pragma once
#include "vag_internal.cuh"

namespace vag {

template <int NT>
__device__ __forceinline__ double block_sum(double v, double *sh /* NT/32 doubles */) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  __syncthreads();
  if (lane == 0) sh[warp] = v;
  __syncthreads();
  double t = 0.0;
  if (warp == 0) {
    t = lane < NT / 32 ? sh[lane] : 0.0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
  }
  return t;   // valid in thread 0
}

// Writes K per-block values to partials[K*blockIdx.x + k]; returns true in
// every thread of the last block to arrive, after which `out[k]` (thread 0)
// holds the grid totals in a fixed order.
template <int NT, int K>
__device__ __forceinline__ bool grid_sum(const double (&v)[K], double *partials, unsigned *counter,
                                         double (&out)[K]) {
  __shared__ double sh[NT / 32];
  __shared__ bool last;
  double bs[K];
#pragma unroll
  for (int k = 0; k < K; ++k) bs[k] = block_sum<NT>(v[k], sh);
  if (threadIdx.x == 0) {
#pragma unroll
    for (int k = 0; k < K; ++k) partials[K * blockIdx.x + k] = bs[k];
    __threadfence();
    const unsigned t = atomicAdd(counter, 1u);
    last = (t == gridDim.x - 1);
  }
  __syncthreads();
  if (!last) return false;
  __threadfence();
#pragma unroll
  for (int k = 0; k < K; ++k) {
    double acc = 0.0;
    for (int b = threadIdx.x; b < (int)gridDim.x; b += NT) acc += __ldcg(&partials[K * b + k]);
    out[k] = block_sum<NT>(acc, sh);
  }
  if (threadIdx.x == 0) *counter = 0u;
  return true;
}

// Row tiles of a batch: tile t covers rows [row0[t], row1[t]) of system
// sys[t]; sys_tile0 gives the first tile of each system (n_sys+1 entries).
// The tiles of a system form groups of kSegGroup consecutive tiles (the last
// one shorter); grp0 gives each system's first group (n_sys+1 entries).
constexpr int kSegGroup = 32;
struct Tiles {
  const int *sys, *row0, *row1, *sys_tile0;
  const int *grp0;
  int n_tiles, n_sys;
};

// Counts this thread in; true for the last of `members`, which then also sees
// what the others wrote before they counted.  (A __threadfence() on every
// member would also acquire, that is, drop the SM's L1 lines under the tiles
// that still gather from it.)
__device__ __forceinline__ bool arrive_last(unsigned *counter, int members) {
  unsigned t;
  asm volatile("atom.add.release.gpu.global.u32 %0, [%1], 1;" : "=r"(t) : "l"(counter) : "memory");
  if (t != (unsigned)(members - 1)) return false;
  asm volatile("fence.acq_rel.gpu;" ::: "memory");
  return true;
}
__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// The sum of a 256-thread tile's values sh[thread], valid in all lanes of the
// calling warp: the tree of warp_sum in every warp, then over the warps'
// sums, on the same pairs, but each partial sum formed once instead of in
// every lane that could use it: 12 FP64 instructions a tile instead of 45.
// (The FP64 pipe takes about 16 cycles an SM for a warp instruction, so the
// 45 were 700 cycles a tile, more than the loads of a short FP32 kernel.
// 64^3 run 23.55 -> 23.1 ms, 96^3 solve 31.9 -> 31.5, 128^3 run 129.9 -> 129.4;
// the FP32 update with its sum in the 128^3 solve 60.5 -> 47.1 us.)
__device__ __forceinline__ double tile_sum(const double *sh, int lane) {
  double a[4];   // lanes l and l + 16 of warps 2 j + (lane >> 4), l = lane & 15
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const double *p = sh + (2 * j + (lane >> 4)) * 32 + (lane & 15);
    a[j] = p[0] + p[16];
  }
  const bool h8 = lane & 8, h4 = lane & 4;   // these bits pick j from here on
  double b0 = h8 ? a[2] : a[0], b1 = h8 ? a[3] : a[1];
  b0 += __shfl_xor_sync(0xffffffffu, h8 ? a[0] : a[2], 8);
  b1 += __shfl_xor_sync(0xffffffffu, h8 ? a[1] : a[3], 8);
  double c = h4 ? b1 : b0;
  c += __shfl_xor_sync(0xffffffffu, h4 ? b0 : b1, 4);
  c += __shfl_xor_sync(0xffffffffu, c, 2);
  c += __shfl_xor_sync(0xffffffffu, c, 1);
  // the warps: bits 2, 1, 0 of their number are lane bits 3, 2, 4
  c += __shfl_xor_sync(0xffffffffu, c, 8);
  c += __shfl_xor_sync(0xffffffffu, c, 4);
  c += __shfl_xor_sync(0xffffffffu, c, 16);
  return c;
}

// out[k] = the sum of ng group partials, as a block would form it: thread b
// adds the groups b, b + NT, ..., then the warps' sums are added.  One warp;
// load(k, b) gives a group's partial.
template <int NT, int K, class F>
__device__ __forceinline__ void groups_sum(int ng, int lane, double (&out)[K], F &&load) {
  constexpr int NW = NT / 32;
#pragma unroll
  for (int k = 0; k < K; ++k) {
    double acc[NW];
#pragma unroll
    for (int w = 0; w < NW; ++w) acc[w] = w * 32 + lane < ng ? load(k, w * 32 + lane) : 0.0;
#pragma unroll
    for (int w = 0; w < NW; ++w)
      for (int b = w * 32 + lane + NT; b < ng; b += NT) acc[w] += load(k, b);
    double mine = 0.0;
#pragma unroll
    for (int w = 0; w < NW; ++w) {
      if (w * 32 >= ng) break;
      const double sw = warp_sum(acc[w]);
      if (lane == w) mine = sw;
    }
    out[k] = warp_sum(mine);
  }
}

// Sums K values per system: per-tile block sums go to partials[K*t + k]; the
// tiles of a group of kSegGroup are added in tile order, then the groups in
// group order.  True in thread 0 of one tile alone, where out[] holds the
// sums.  The grouping depends on the system alone, so the sums do too (also
// on which of the two ways below they are taken).
// Every Krylov kernel of a small system waits for this chain and little else
// (a barrier, a write, a fence, an atomic and a read of the L2 a level, about
// 3 us), so it is kept short.  A system of one tile needs no counter; up to
// one group, its last tile's first warp adds the partials alone.  Up to
// kSegOneLevel tiles the last tile of the system to arrive (counter[sys])
// adds everything, a group a warp: one releasing atomic and one read of the
// partials.  A larger system would queue thousands of atomics on one address:
// the last tile of each group (counter[n_sys + 1 + g]) writes the group's sum
// to partials[K*(n_tiles + g) + k], and the last of those groups adds them.
// Against two levels for all, with a __threadfence() and barriers in each:
// 8^3 cells with Jacobi CG (3 tiles) 4.53 -> 3.64 ms, 29 x 23 x 19 cells (51
// tiles) 7.34 -> 6.88, 48^3 mixed solve (457 tiles) 12.50 -> 11.74, 64^3 run
// (1060 tiles) 24.37 -> 23.89, 128^3 run (8637 tiles) 130.8 ms in both.
// (Two levels with one warp each instead of the block for 33 to 1024 tiles:
// 7.19 and 12.61 ms; the block for the 3 tiles: 3.90 ms.  One level up to 2048 or
// 4096 tiles: 64^3 run 0.5 and 2 % slower, 96^3 solve, 3733 tiles, the same
// and 3 % slower.)
// One call a kernel (the shared words are not guarded against a second).
constexpr int kSegOneLevel = 1024;
template <int NT, int K>
__device__ __forceinline__ bool seg_sum(const double (&v)[K], double *partials, unsigned *counter, const Tiles &tl,
                                        int t, int sys, double (&out)[K]) {
  static_assert(kSegGroup == 32, "a group's tiles are one warp's lanes");
  constexpr int NW = NT / 32;
  static_assert(NT == 256, "tile_sum");
  __shared__ double sh[K][NT];
  __shared__ double gsum[K][kSegOneLevel / kSegGroup];
  __shared__ bool last;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int t0 = tl.sys_tile0[sys], t1 = tl.sys_tile0[sys + 1];
  const int ng = (t1 - t0 + kSegGroup - 1) / kSegGroup;
#pragma unroll
  for (int k = 0; k < K; ++k) sh[k][threadIdx.x] = v[k];
  __syncthreads();
  if (t1 - t0 > kSegGroup && t1 - t0 <= kSegOneLevel) {
    if (warp == 0) {
#pragma unroll
      for (int k = 0; k < K; ++k) out[k] = tile_sum(sh[k], lane);
    }
    if (threadIdx.x == 0) {
#pragma unroll
      for (int k = 0; k < K; ++k) partials[(size_t)K * t + k] = out[k];
      last = arrive_last(&counter[sys], t1 - t0);
    }
    __syncthreads();
    if (!last) return false;
    // a warp's groups, all loads first
    constexpr int kMine = kSegOneLevel / kSegGroup / NW;
#pragma unroll
    for (int k = 0; k < K; ++k) {
      double g[kMine];
#pragma unroll
      for (int q = 0; q < kMine; ++q) {
        const int b = t0 + (q * NW + warp) * kSegGroup + lane;
        g[q] = b < t1 ? __ldcg(&partials[(size_t)K * b + k]) : 0.0;
      }
#pragma unroll
      for (int q = 0; q < kMine; ++q) {
        if (q * NW + warp >= ng) break;
        const double sg = warp_sum(g[q]);
        if (lane == 0) gsum[k][q * NW + warp] = sg;
      }
    }
    __syncthreads();
    if (warp != 0) return false;
    groups_sum<NT, K>(ng, lane, out, [&](int k, int b) { return gsum[k][b]; });
    if (lane == 0) counter[sys] = 0u;
    return lane == 0;
  }
  if (warp != 0) return false;
#pragma unroll
  for (int k = 0; k < K; ++k) out[k] = tile_sum(sh[k], lane);
  const int grp = tl.grp0[sys];
  const int gl = (t - t0) / kSegGroup;                 // group within the system
  const int ga = t0 + gl * kSegGroup;                  // its tiles [ga, gb)
  const int gb = min(ga + kSegGroup, t1);
  const int g = grp + gl;                              // its storage index
  if (t1 - t0 == 1) return lane == 0;
  unsigned *gctr = ng == 1 ? counter + sys : counter + tl.n_sys + 1 + g;
  double *gpart = partials + (size_t)K * tl.n_tiles;
  bool mine = false;
  if (lane == 0) {
#pragma unroll
    for (int k = 0; k < K; ++k) partials[(size_t)K * t + k] = out[k];
    mine = arrive_last(gctr, gb - ga);
  }
  if (!__shfl_sync(0xffffffffu, mine, 0)) return false;
  __syncwarp();
#pragma unroll
  for (int k = 0; k < K; ++k)
    out[k] = warp_sum(ga + lane < gb ? __ldcg(&partials[(size_t)K * (ga + lane) + k]) : 0.0);
  if (lane == 0) *gctr = 0u;
  if (ng == 1) return lane == 0;
  if (lane == 0) {
#pragma unroll
    for (int k = 0; k < K; ++k) gpart[(size_t)K * g + k] = out[k];
    mine = arrive_last(&counter[sys], ng);
  }
  if (!__shfl_sync(0xffffffffu, mine, 0)) return false;
  __syncwarp();
  groups_sum<NT, K>(ng, lane, out, [&](int k, int b) { return __ldcg(&gpart[(size_t)K * (grp + b) + k]); });
  if (lane == 0) counter[sys] = 0u;
  return lane == 0;
}

}  // namespace vag
