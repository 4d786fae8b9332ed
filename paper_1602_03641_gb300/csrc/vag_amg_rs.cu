// Classical (Ruge-Stueben-type) coarsening for the AMG hierarchy: the
// counterpart of the classical AMG (Hypre's BoomerAMG) that the paper's
// solver experiments (Sec. 5.3-5.4) found robust in the fracture/matrix
// permeability ratio.  Written from the classical construction (Ruge and
// Stueben, "Algebraic multigrid", 1987; Stueben, "A review of algebraic
// multigrid", 2001) with the parallel PMIS splitting (De Sterck, Yang, Heys,
// SIAM J. Matrix Anal. Appl. 27, 2006).  Per level, all on the device:
//  strength   i depends strongly on j != i when -a_ij >= theta max_{k != i}
//             (-a_ik) (negative couplings; positive ones never count);
//  measure    the number of rows that depend strongly on i; the eliminated
//             VAG matrix is symmetric, so whether j depends on i is read from
//             row i's entry a_ij and row j's largest negative coupling, with
//             no transpose of the strength graph;
//  PMIS       rows no row depends on are fine from the start; then, in
//             rounds, an undecided row whose key (measure, a hash of its
//             system-local index, the index) is the largest among its
//             undecided strong neighbours (either direction) becomes coarse,
//             and undecided rows that depend on a new coarse row become fine;
//  2nd pass   a fine row with strong connections but no coarse one becomes
//             coarse, so every such row interpolates from at least one;
//  P          direct interpolation: coarse rows copy their value; a fine row
//             i takes w_ij = -alpha_i a_ij / (a_ii + sum_{k != i} a_ik^+) from
//             its strong coarse neighbours (at most kPmax, the largest
//             |a_ij|, ties by index), alpha_i = (sum of all its negative
//             couplings) / (sum over the chosen ones), so that P maps the
//             constant to the constant on zero-row-sum rows; rows without
//             strong connections interpolate from nothing (the smoother
//             handles them);
//  R = P^T    transposed with its rows sorted by fine index;
//  Galerkin   A_c = R A P, one coarse row per warp, every entry summed in a
//             fixed sequence order and the row's columns in the order they
//             first appear (deterministic: a system's hierarchy depends on
//             that system alone, so it is bitwise the same in a batch).
#include <climits>
#include <functional>
#include <vector>

#include "vag_internal.cuh"

namespace vag {
namespace {

constexpr int TB = 256;
constexpr double kRsTheta = 0.25;
constexpr int kPmax = 4;
constexpr int kMaxRounds = 64;

__device__ __forceinline__ uint32_t rs_hash(uint32_t x) {
  x ^= x >> 16; x *= 0x7feb352dU; x ^= x >> 15; x *= 0x846ca68bU; x ^= x >> 16;
  return x;
}

__device__ __forceinline__ int rs_sys_of_row(int i, const int *__restrict__ start, int n_sys) {
  int lo = 0, hi = n_sys - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (start[mid] <= i) lo = mid; else hi = mid - 1;
  }
  return lo;
}

// How the setup kernels walk a level's rows: LN lanes per row, lane l taking
// its entries l, l + LN, ...; entry k of row i is at p0 + k stride.
//  LN = 1, the finest level in its sliced ELL: 32 rows of a warp read entry k
//          as one segment (in CSR, a thread per row touched 32 lines a load:
//          maxneg to p_fill took 3.0 ms at 128^3);
//  LN = 8, coarse levels in CSR: their rows of 40 entries are read in 64-byte
//          segments, and a level of a few thousand rows, where a thread's
//          serial walk of its row was all the time (60-110 us a kernel
//          whatever the level's size), takes a fifth of it.
template <int LN>
struct Rows {
  int n;
  const int *rowptr, *slice_ptr, *col;
  const double *val;
  __device__ __forceinline__ int len(int i) const { return rowptr[i + 1] - rowptr[i]; }
  __device__ __forceinline__ int first(int i) const {
    return LN == 1 ? slice_ptr[i >> 5] + (i & 31) : rowptr[i];
  }
  static constexpr int stride = LN == 1 ? 32 : 1;
  // row of this thread (n or more: none) and its lane in the row
  static __device__ __forceinline__ int row() { return (int)((blockIdx.x * (unsigned)TB + threadIdx.x) / LN); }
  static __device__ __forceinline__ int lane() { return threadIdx.x & (LN - 1); }
};
// combine over the lanes of a row (every lane of the warp calls it)
template <int LN, class T, class F>
__device__ __forceinline__ T over_lanes(T v, F &&f) {
#pragma unroll
  for (int o = LN / 2; o >= 1; o /= 2) v = f(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

// largest negative coupling -a_ik over k != i (0 when there is none)
template <int LN>
__global__ void __launch_bounds__(TB) k_rs_maxneg(Rows<LN> A, double *__restrict__ maxneg) {
  const int i = A.row(), l = A.lane();
  double m = 0.0;
  if (i < A.n) {
    const int len = A.len(i), p0 = A.first(i);
    for (int k = l; k < len; k += LN) {
      const int p = p0 + k * A.stride;
      const double a = -A.val[p];
      if (A.col[p] != i && a > m) m = a;
    }
  }
  m = over_lanes<LN>(m, [](double x, double y) { return x > y ? x : y; });
  if (i < A.n && l == 0) maxneg[i] = m;
}

// i depends strongly on j through the entry a (= a_ij = a_ji)
__device__ __forceinline__ bool rs_strong(double a, double maxneg_row) {
  return maxneg_row > 0.0 && -a >= kRsTheta * maxneg_row;
}

// state: 0 undecided, 1 coarse, -1 fine, -2 fine without strong connections
// (interpolates from nothing), -3 row of a system solved densely here
template <int LN>
__global__ void __launch_bounds__(TB) k_rs_init(Rows<LN> A, const double *__restrict__ maxneg,
                                                const uint8_t *__restrict__ skip, const int *__restrict__ sys_start,
                                                int n_sys, unsigned long long *__restrict__ key,
                                                int8_t *__restrict__ state, uint8_t *__restrict__ sflag) {
  const int i = A.row(), l = A.lane();
  const bool valid = i < A.n;
  const bool sk = valid && skip[i];
  int depends = 0, infl = 0;
  if (valid) {
    const int len = A.len(i), p0 = A.first(i);
    const double mi = maxneg[i];
    for (int k = l; k < len; k += LN) {
      const int p = p0 + k * A.stride, j = A.col[p];
      uint8_t f = 0;
      if (j != i && !sk) {
        const double a = A.val[p];
        const bool dij = rs_strong(a, mi);          // i depends on j
        const bool dji = rs_strong(a, maxneg[j]);   // j depends on i
        depends |= dij;
        infl += dji;
        f = (uint8_t)(dij | (dji << 1));
      }
      sflag[p] = f;   // the strength of the entry, both ways, for the PMIS rounds
    }
  }
  depends = over_lanes<LN>(depends, [](int x, int y) { return x | y; });
  infl = over_lanes<LN>(infl, [](int x, int y) { return x + y; });
  if (!valid || l != 0) return;
  if (sk) {
    key[i] = 0;
    state[i] = -3;
    return;
  }
  const int loc = i - sys_start[rs_sys_of_row(i, sys_start, n_sys)];
  key[i] = ((unsigned long long)(infl < 65535 ? infl : 65535) << 48) |
           ((unsigned long long)(rs_hash((uint32_t)loc) & 0xffffu) << 32) | (uint32_t)loc;
  state[i] = (!depends && infl == 0) ? -2 : (infl == 0 ? -1 : 0);
}

// PMIS round, first half: undecided rows that are the largest among their
// undecided strong neighbours become coarse
template <int LN>
__global__ void __launch_bounds__(TB) k_rs_pmis_c(Rows<LN> A, const uint8_t *__restrict__ sflag,
                                                  const unsigned long long *__restrict__ key,
                                                  const int8_t *__restrict__ st_in, int8_t *__restrict__ st_out,
                                                  int *undecided) {
  const int i = A.row(), l = A.lane();
  if (i == 0 && l == 0) *undecided = 0;   // counted by the round's second half
  const int8_t s = i < A.n ? st_in[i] : (int8_t)1;
  int top = 1;
  if (s == 0) {
    const unsigned long long ki = key[i];
    const int len = A.len(i), p0 = A.first(i);
    for (int k = l; k < len && top; k += LN) {
      const int p = p0 + k * A.stride;
      if (!sflag[p]) continue;   // not strong either way (or the diagonal)
      const int j = A.col[p];
      if (st_in[j] == 0 && key[j] > ki) top = 0;
    }
  }
  top = over_lanes<LN>(top, [](int x, int y) { return x & y; });
  if (i < A.n && l == 0) st_out[i] = s != 0 ? s : (int8_t)top;
}

// second half: undecided rows that depend on a coarse row become fine; the
// rest are counted
template <int LN>
__global__ void __launch_bounds__(TB) k_rs_pmis_f(Rows<LN> A, const uint8_t *__restrict__ sflag,
                                                  const int8_t *__restrict__ st_in, int8_t *__restrict__ st_out,
                                                  int *undecided) {
  const int i = A.row(), l = A.lane();
  const int8_t s = i < A.n ? st_in[i] : (int8_t)1;
  int fine = 0;
  if (s == 0) {
    const int len = A.len(i), p0 = A.first(i);
    for (int k = l; k < len && !fine; k += LN) {
      const int p = p0 + k * A.stride;
      fine = (sflag[p] & 1) && st_in[A.col[p]] == 1;   // i depends on a coarse row
    }
  }
  fine = over_lanes<LN>(fine, [](int x, int y) { return x | y; });
  if (i < A.n && l == 0) st_out[i] = s != 0 ? s : (int8_t)-fine;
  // one atomic per warp for the rows still undecided
  const unsigned m = __ballot_sync(0xffffffffu, l == 0 && s == 0 && !fine);
  if ((threadIdx.x & 31) == 0 && m) atomicAdd(undecided, __popc(m));
}

// second pass: a fine row that depends on rows but on no coarse one becomes
// coarse
template <int LN>
__global__ void __launch_bounds__(TB) k_rs_second_pass(Rows<LN> A, const uint8_t *__restrict__ sflag,
                                                       const int8_t *__restrict__ st_in, int8_t *__restrict__ st_out,
                                                       int *__restrict__ cflag) {
  const int i = A.row(), l = A.lane();
  int8_t s = i < A.n ? st_in[i] : (int8_t)1;
  int has = 0;   // 1: depends on some row, 2: on a coarse one
  if (s == -1) {
    const int len = A.len(i), p0 = A.first(i);
    for (int k = l; k < len; k += LN) {
      const int p = p0 + k * A.stride;
      if (sflag[p] & 1) has |= st_in[A.col[p]] == 1 ? 3 : 1;
    }
  }
  has = over_lanes<LN>(has, [](int x, int y) { return x | y; });
  if (i >= A.n || l != 0) return;
  if (has == 1) s = 1;
  st_out[i] = s;
  cflag[i] = s == 1;
}

// P's row i before the coarse numbering is known: the entries it takes (a
// coarse row: itself; a fine row: its strong coarse neighbours, at most kPmax
// of them with the largest |a_ij|, ties by position) as positions in the
// level's entry array, in row order, and (alpha_i, a_ii + sum of the positive
// couplings), the sums taken in row order whatever LN.
template <int LN>
__global__ void __launch_bounds__(TB) k_rs_choose(Rows<LN> A, const uint8_t *__restrict__ sflag,
                                                  const int8_t *__restrict__ st, int *__restrict__ cnt,
                                                  int4 *__restrict__ picks, double2 *__restrict__ factor,
                                                  int *status) {
  static_assert(kPmax == 4, "picks of a row are one int4");
  const int i = A.row(), l = A.lane();
  const int8_t s = i < A.n ? st[i] : (int8_t)0;
  double aii = 0.0, neg = 0.0, pos = 0.0;
  int pk[kPmax];
  double pa[kPmax];
  int m = 0;
  const int len = s == -1 ? A.len(i) : 0, p0 = s == -1 ? A.first(i) : 0;
  const int rounds = LN == 1 ? len : __reduce_max_sync(0xffffffffu, (len + LN - 1) / LN);
  for (int k = l, round = 0; round < rounds; ++round, k += LN) {
    double a = 0.0;
    int kind = 3;   // 0 diagonal, 1 negative, 2 positive coupling, 3 none
    if (k < len) {
      const int p = p0 + k * A.stride, j = A.col[p];
      a = A.val[p];
      kind = j == i ? 0 : a < 0.0 ? 1 : 2;
      if ((sflag[p] & 1) && st[j] == 1 && !(m == kPmax && !(a < pa[kPmax - 1]))) {
        // into this lane's kPmax strongest (a < 0: the smallest values), strongest first
        int q = m < kPmax ? m++ : kPmax - 1;
#pragma unroll
        for (int t = kPmax - 1; t > 0; --t)
          if (t == q) {
            if (!(a < pa[t - 1])) {
              pk[t] = k;
              pa[t] = a;
              q = -1;
            } else {
              pk[t] = pk[t - 1];
              pa[t] = pa[t - 1];
              q = t - 1;
            }
          }
        if (q == 0) {
          pk[0] = k;
          pa[0] = a;
        }
      }
    }
#pragma unroll
    for (int t = 0; t < LN; ++t) {   // the lanes' entries in row order
      const double at = LN == 1 ? a : __shfl_sync(0xffffffffu, a, t, LN);
      const int kt = LN == 1 ? kind : __shfl_sync(0xffffffffu, kind, t, LN);
      if (kt == 0) aii += at;
      else if (kt == 1) neg += at;
      else if (kt == 2) pos += at;
    }
  }
  double cneg = 0.0;
  if (LN > 1) {
    // the row's kPmax strongest from the lanes' lists: kPmax rounds of the
    // strongest head (ties by position)
    int gk[kPmax], gm = 0;
    double ga[kPmax];
#pragma unroll
    for (int t = 0; t < kPmax; ++t) {
      double ba = m > 0 ? pa[0] : 0.0;
      int bk = m > 0 ? pk[0] : INT_MAX;
#pragma unroll
      for (int o = LN / 2; o >= 1; o /= 2) {
        const double oa = __shfl_xor_sync(0xffffffffu, ba, o);
        const int ok = __shfl_xor_sync(0xffffffffu, bk, o);
        if (oa < ba || (oa == ba && ok < bk)) { ba = oa; bk = ok; }
      }
      gk[t] = bk;
      ga[t] = ba;
      if (bk != INT_MAX) {
        gm = t + 1;
        if (m > 0 && pk[0] == bk) {   // taken from this lane's list
#pragma unroll
          for (int u = 0; u + 1 < kPmax; ++u) { pk[u] = pk[u + 1]; pa[u] = pa[u + 1]; }
          --m;
        }
      }
    }
    m = gm;
#pragma unroll
    for (int t = 0; t < kPmax; ++t) { pk[t] = gk[t]; pa[t] = ga[t]; }
  }
  if (i >= A.n || l != 0) return;
  if (s != -1) {
    cnt[i] = s == 1;
    return;
  }
  // row order
#pragma unroll
  for (int p = 1; p < kPmax; ++p)
#pragma unroll
    for (int q = p; q > 0; --q)
      if (p < m && pk[q - 1] > pk[q]) {
        const int t = pk[q]; pk[q] = pk[q - 1]; pk[q - 1] = t;
        const double x = pa[q]; pa[q] = pa[q - 1]; pa[q - 1] = x;
      }
#pragma unroll
  for (int q = 0; q < kPmax; ++q)
    if (q < m) cneg += pa[q];
  const double diag = aii + pos;
  if (!(diag > 0.0) || !(cneg < 0.0)) {
    atomicOr(status, ST_NONPOSITIVE);
    m = 0;
  }
  int4 o;
  o.x = m > 0 ? p0 + pk[0] * A.stride : 0;
  o.y = m > 1 ? p0 + pk[1] * A.stride : 0;
  o.z = m > 2 ? p0 + pk[2] * A.stride : 0;
  o.w = m > 3 ? p0 + pk[3] * A.stride : 0;
  picks[i] = o;
  factor[i] = make_double2(neg / cneg, diag);
  cnt[i] = m;
}

// P's rows, and R's row counts
__global__ void k_rs_p_fill(int n, const int *__restrict__ acol, const double *__restrict__ aval,
                            const int8_t *__restrict__ st, const int *__restrict__ cidx, const int4 *__restrict__ picks,
                            const double2 *__restrict__ factor, const int *__restrict__ prow, int *__restrict__ pcol,
                            double *__restrict__ pval, int *rcnt) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int o = prow[i], m = prow[i + 1] - o;
  if (m == 0) return;
  if (st[i] == 1) {
    const int I = cidx[i];
    pcol[o] = I;
    pval[o] = 1.0;
    atomicAdd(&rcnt[I], 1);
    return;
  }
  const int4 pk = picks[i];
  const double alpha = factor[i].x, diag = factor[i].y;
  const int p[kPmax] = {pk.x, pk.y, pk.z, pk.w};
#pragma unroll
  for (int q = 0; q < kPmax; ++q)
    if (q < m) {
      const int I = cidx[acol[p[q]]];
      pcol[o + q] = I;
      pval[o + q] = -alpha * aval[p[q]] / diag;
      atomicAdd(&rcnt[I], 1);
    }
}

// R = P^T: entries placed by an atomic cursor, then each row sorted by fine
// index (so its content does not depend on the order of the atomics)
__global__ void k_rs_r_fill(int n, const int *__restrict__ prow, const int *__restrict__ pcol,
                            const double *__restrict__ pval, const int *__restrict__ rrow, int *cursor,
                            int *__restrict__ rcol, double *__restrict__ rval) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  for (int k = prow[i]; k < prow[i + 1]; ++k) {
    const int I = pcol[k];
    const int q = rrow[I] + atomicAdd(&cursor[I], 1);
    rcol[q] = i;
    rval[q] = pval[k];
  }
}

// One warp per row of R, entries in registers, their places by counting the
// smaller indices of the row (rows of up to 32 entries; longer ones, which
// direct interpolation hardly makes, by insertion in one lane).
__global__ void __launch_bounds__(TB) k_rs_r_sort(int nc, const int *__restrict__ rrow, int *rcol, double *rval) {
  const int I = blockIdx.x * (TB / 32) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (I >= nc) return;   // whole warps
  const int b = rrow[I], m = rrow[I + 1] - b;
  if (m <= 32) {
    const int c = lane < m ? rcol[b + lane] : INT_MAX;
    const double v = lane < m ? rval[b + lane] : 0.0;
    int rank = 0;
    for (int q = 0; q < m; ++q) rank += __shfl_sync(0xffffffffu, c, q) < c;
    if (lane < m) {   // every lane has read its entry (the shuffles above)
      rcol[b + rank] = c;
      rval[b + rank] = v;
    }
    return;
  }
  if (lane != 0) return;
  for (int p = b + 1; p < b + m; ++p) {
    const int c = rcol[p];
    const double v = rval[p];
    int q = p - 1;
    while (q >= b && rcol[q] > c) {
      rcol[q + 1] = rcol[q];
      rval[q + 1] = rval[q];
      --q;
    }
    rcol[q + 1] = c;
    rval[q + 1] = v;
  }
}

// A_c = R A P row by row, each warp taking coarse rows I, I + (warps in the
// grid), ...: for every entry r_Ii of row I of R (in order), the entries a_ik
// of row i of A 32 at a time, each lane walking row k of P (at most kPmax
// entries) one entry per round; the contributions r_Ii a_ik p_kJ meet in a
// shared-memory hash keyed by J, lanes that hit the same slot are grouped
// and the lowest adds their values in lane order, so every entry is summed in
// the order (entry of R, chunk of A's row, entry of P, lane), fixed by the
// data.  A column enters the row's list when it first appears, the columns
// new in one round in the order of their lowest lane (a ballot prefix), so
// the list order is fixed by the data too.  A row may use at most HASH/2
// slots (ST_ROW_OVERFLOW otherwise).  Its (column, sum) pairs are written in
// list order to the row's padded slot zcol/zval[I*HASH/2 ..], the table is
// cleared through the list, the count goes to zcnt[I] and 1/z_II to zdinv;
// k_rs_compact packs the rows.
template <int HASH, int WARPS>
__global__ void __launch_bounds__(32 * WARPS) k_rs_rap(int nrows, const int *__restrict__ rrow,
                                                       const int *__restrict__ rcol, const double *__restrict__ rval,
                                                       const int *__restrict__ arow, const int *__restrict__ acol,
                                                       const double *__restrict__ aval,
                                                       const int *__restrict__ prow, const int *__restrict__ pcol,
                                                       const double *__restrict__ pval, int *__restrict__ zcnt,
                                                       int *__restrict__ zcol, double *__restrict__ zval,
                                                       double *__restrict__ zdinv, int *status) {
  constexpr int CAP = HASH / 2;
  __shared__ int keys[WARPS][HASH];
  __shared__ double sums[WARPS][HASH];
  __shared__ int used[WARPS][CAP];
  __shared__ double vals[WARPS][32];
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const unsigned below = (1u << lane) - 1u;
  int *K = keys[w];
  double *S = sums[w];
  int *U = used[w];
  for (int h = lane; h < HASH; h += 32) {
    K[h] = -1;
    S[h] = 0.0;
  }
  __syncwarp();
  const int stride = gridDim.x * WARPS;
  for (int I = blockIdx.x * WARPS + w; I < nrows; I += stride) {   // a whole warp takes each row
    int nu = 0;                 // columns listed so far (the same in every lane)
    bool overflow = false;
    // one round: each lane offers (J, v) (J < 0: nothing)
    auto add = [&](int J, double v) {
      int slot = -1;
      bool claimed = false;
      if (J >= 0) {
        unsigned h = ((unsigned)J * 2654435761u) & (HASH - 1);
        for (int probe = 0; probe < HASH; ++probe, h = (h + 1) & (HASH - 1)) {
          const int cur = ((volatile int *)K)[h];
          if (cur == J) { slot = (int)h; break; }
          if (cur == -1) {
            const int old = atomicCAS(&K[h], -1, J);
            if (old == -1) { slot = (int)h; claimed = true; break; }
            if (old == J) { slot = (int)h; break; }
          }
        }
        if (slot < 0) overflow = true;
      }
      vals[w][lane] = v;
      __syncwarp();
      const unsigned grp = __match_any_sync(0xffffffffu, slot >= 0 ? slot : -1 - lane);
      const bool is_new = (grp & __ballot_sync(0xffffffffu, claimed)) != 0;
      const bool leader = slot >= 0 && lane == __ffs(grp) - 1;
      const unsigned lead_new = __ballot_sync(0xffffffffu, leader && is_new);
      if (leader && is_new) {
        const int q = nu + __popc(lead_new & below);
        if (q < CAP) U[q] = slot;
      }
      nu += __popc(lead_new);
      if (leader) {
        double acc = S[slot];
        for (unsigned m = grp; m; m &= m - 1) acc += vals[w][__ffs(m) - 1];
        S[slot] = acc;
      }
      __syncwarp();
    };
    for (int kr = rrow[I]; kr < rrow[I + 1]; ++kr) {
      const int i = rcol[kr];
      const double r = rval[kr];
      const int ab = arow[i], ae = arow[i + 1];
      for (int c = ab; c < ae; c += 32) {
        const int k = c + lane;
        int eb = 0, len = 0;
        double a = 0.0;
        if (k < ae) {
          const int j = acol[k];
          a = r * aval[k];
          eb = prow[j];
          len = prow[j + 1] - eb;
        }
        const int mlen = __reduce_max_sync(0xffffffffu, len);
        for (int e = 0; e < mlen; ++e) add(e < len ? pcol[eb + e] : -1, e < len ? a * pval[eb + e] : 0.0);
      }
    }
    __syncwarp();
    const bool bad = __any_sync(0xffffffffu, overflow) || nu > CAP;
    if (bad) {
      if (lane == 0) {
        atomicOr(status, ST_ROW_OVERFLOW);
        zcnt[I] = 0;
      }
      // the list is incomplete: clear the whole table
      for (int h = lane; h < HASH; h += 32) {
        K[h] = -1;
        S[h] = 0.0;
      }
      __syncwarp();
      continue;
    }
    if (lane == 0) zcnt[I] = nu;
    const size_t base = (size_t)I * CAP;   // the row's padded slot; compacted afterwards
    bool diag = false;
    for (int q = lane; q < nu; q += 32) {
      const int h = U[q];
      const int J = K[h];
      const double z = S[h];
      zcol[base + q] = J;
      zval[base + q] = z;
      K[h] = -1;
      S[h] = 0.0;
      if (zdinv && J == I) {
        diag = true;
        if (!(z > 0.0)) atomicOr(status, ST_NONPOSITIVE);
        zdinv[I] = 1.0 / z;
      }
    }
    if (zdinv && !__any_sync(0xffffffffu, diag) && lane == 0) {
      atomicOr(status, ST_NONPOSITIVE);
      zdinv[I] = 1.0 / 0.0;
    }
    __syncwarp();
  }
}

// grids of k_rs_rap: enough warps to fill the GPU a few times over, each
// warp then walks many rows
static int rap_blocks(int nrows, int warps) {
  const int want = (nrows + warps - 1) / warps;
  const int cap = num_sms() * 32;
  return std::max(1, std::min(want, cap));
}

// Pack the rows, one warp per row (a row a thread: 1.0 ms of the 128^3 setup).
template <int CAP>
__global__ void __launch_bounds__(TB) k_rs_compact(int nc, const int *__restrict__ tcol,
                                                   const double *__restrict__ tval, const int *__restrict__ rowptr,
                                                   int *__restrict__ col, double *__restrict__ val) {
  const int I = blockIdx.x * (TB / 32) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (I >= nc) return;
  const size_t base = (size_t)I * CAP;
  const int o = rowptr[I], m = rowptr[I + 1] - o;
  for (int q = lane; q < m; q += 32) {
    col[o + q] = tcol[base + q];
    val[o + q] = tval[base + q];
  }
}

__global__ void k_rs_coarse_starts(int n_sys, const int *__restrict__ sys_start, const int *__restrict__ cscan,
                                   int *csys_start) {
  const int g = blockIdx.x * blockDim.x + threadIdx.x;
  if (g <= n_sys) csys_start[g] = cscan[sys_start[g]];
}

// stream-ordered temporaries of the context's pool, freed on every path
struct RsTemps {
  Ctx *c;
  std::vector<void *> p;
  ~RsTemps() {
    for (void *q : p) ctx_free(c, q);
  }
  void *operator()(size_t bytes) {
    void *q = ctx_alloc(c, bytes ? bytes : 1);
    p.push_back(q);
    return q;
  }
};

}  // namespace

void rs_coarsen(System *s, AmgLevel &L, AmgLevel &C, const std::function<void *(size_t)> &alloc) {
  cudaStream_t st = s->ctx->stream;
  const int n = L.n, ns = s->seg.n_sys;
  RsTemps tmp{s->ctx, {}};
  trace_mark(st, "  classical: enter");
  double *maxneg = static_cast<double *>(tmp(8 * (size_t)std::max(n, 1)));
  unsigned long long *key = static_cast<unsigned long long *>(tmp(8 * (size_t)std::max(n, 1)));
  int8_t *sa = static_cast<int8_t *>(tmp(std::max(n, 1)));
  int8_t *sb = static_cast<int8_t *>(tmp(std::max(n, 1)));
  int *undecided = static_cast<int *>(tmp(sizeof(int)));
  const int g = grid_for(n, TB);
  // the finest level (the system's own matrix) is walked in its sliced ELL
  const bool sell = L.slice_ptr != nullptr;
  const int64_t entries = sell ? L.sell_nnz : L.nnz;
  const int *acol = sell ? L.scol : L.col;
  const double *aval = sell ? L.sval : L.val;
  const Rows<1> A1{n, L.rowptr, L.slice_ptr, acol, aval};
  const Rows<8> A8{n, L.rowptr, nullptr, acol, aval};
  const int ga = sell ? g : grid_for(8 * (int64_t)n, TB);
#define RS_LAUNCH(kernel, ...)                                                       \
  do {                                                                               \
    if (sell) kernel<1><<<ga, TB, 0, st>>>(A1, __VA_ARGS__);                         \
    else kernel<8><<<ga, TB, 0, st>>>(A8, __VA_ARGS__);                              \
    note_launches(1);                                                                \
  } while (0)
  uint8_t *sflag = static_cast<uint8_t *>(tmp((size_t)std::max<int64_t>(entries, 1)));
  VAG_CUDA(cudaMemsetAsync(s->status, 0, sizeof(int), st));   // checked after the Galerkin product
  RS_LAUNCH(k_rs_maxneg, maxneg);
  RS_LAUNCH(k_rs_init, maxneg, L.skip, L.d_sys_start, ns, key, sa, sflag);
  VAG_CHECK_LAUNCH();
  trace_mark(st, "  classical: strength + measure");
  // PMIS rounds (two kernels each, states ping-pong).  The second pass, P's
  // row counts and their scans follow without a wait; one read-back then
  // brings the undecided rows, the coarse count and P's nonzeros (R = P^T has
  // as many), and rows still undecided take four more rounds and the same
  // again (a round after the last decision changes nothing).
  int *pin = ctx_pin(s->ctx);
  int *cflag = static_cast<int *>(tmp(4 * (size_t)std::max(n, 1)));
  int *cidx = static_cast<int *>(tmp(4 * ((size_t)n + 1)));
  int *pcnt = static_cast<int *>(tmp(4 * ((size_t)n + 1)));
  int4 *picks = static_cast<int4 *>(tmp(16 * (size_t)std::max(n, 1)));
  double2 *factor = static_cast<double2 *>(tmp(16 * (size_t)std::max(n, 1)));
  L.prow = static_cast<int *>(alloc(4 * ((size_t)n + 1)));
  const int8_t *state = sb;
  bool finished = false;
  for (int r = 0, next = n > 2000 ? 8 : 4; r < kMaxRounds && !finished; next += 4) {
    for (; r < next; ++r) {
      RS_LAUNCH(k_rs_pmis_c, sflag, key, sa, sb, undecided);
      RS_LAUNCH(k_rs_pmis_f, sflag, sb, sa, undecided);
    }
    trace_mark(st, "  classical: PMIS rounds");
    RS_LAUNCH(k_rs_second_pass, sflag, sa, sb, cflag);
    scan_exclusive(s->ctx, cflag, cidx, n, false);
    RS_LAUNCH(k_rs_choose, sflag, state, pcnt, picks, factor, s->status);
    scan_exclusive(s->ctx, pcnt, L.prow, n, false);
    VAG_CUDA(cudaMemcpyAsync(&pin[0], cidx + n, sizeof(int), cudaMemcpyDeviceToHost, st));
    VAG_CUDA(cudaMemcpyAsync(&pin[1], L.prow + n, sizeof(int), cudaMemcpyDeviceToHost, st));
    VAG_CUDA(cudaMemcpyAsync(&pin[2], undecided, sizeof(int), cudaMemcpyDeviceToHost, st));
    VAG_CUDA(cudaStreamSynchronize(st));
    finished = pin[2] == 0;
    if (!finished) VAG_CUDA(cudaMemsetAsync(s->status, 0, sizeof(int), st));
  }
#undef RS_LAUNCH
  if (!finished) fail(VAG_ECUDA, "AMG: the PMIS splitting did not finish");
  const int nc = pin[0];
  L.p_nnz = pin[1];
  L.pcol = static_cast<int *>(alloc(4 * (size_t)std::max<int64_t>(L.p_nnz, 1)));
  L.pval = static_cast<double *>(alloc(8 * (size_t)std::max<int64_t>(L.p_nnz, 1)));
  // R = P^T (its row counts come with P)
  int *rcnt = static_cast<int *>(tmp(8 * ((size_t)nc + 1)));
  int *cursor = rcnt + nc + 1;
  L.rrow = static_cast<int *>(alloc(4 * ((size_t)nc + 1)));
  VAG_CUDA(cudaMemsetAsync(rcnt, 0, 8 * ((size_t)nc + 1), st));
  k_rs_p_fill<<<g, TB, 0, st>>>(n, acol, aval, state, cidx, picks, factor, L.prow, L.pcol, L.pval, rcnt);
  note_launches(1);
  scan_exclusive(s->ctx, rcnt, L.rrow, nc, false);
  L.r_nnz = L.p_nnz;
  L.rcol = static_cast<int *>(alloc(4 * (size_t)std::max<int64_t>(L.r_nnz, 1)));
  L.rval = static_cast<double *>(alloc(8 * (size_t)std::max<int64_t>(L.r_nnz, 1)));
  k_rs_r_fill<<<g, TB, 0, st>>>(n, L.prow, L.pcol, L.pval, L.rrow, cursor, L.rcol, L.rval);
  k_rs_r_sort<<<grid_for(nc, TB / 32), TB, 0, st>>>(nc, L.rrow, L.rcol, L.rval);
  note_launches(2);
  VAG_CHECK_LAUNCH();
  L.nc = nc;
  trace_mark(st, "  classical: second pass, P, R");
  // Galerkin A_c = R A P in one pass into rows padded to kRapHash/2 columns,
  // then packed
  constexpr int kRapHash = 512, kRapWarps = 4, kRapCap = kRapHash / 2;
  C.n = nc;
  C.rowptr = static_cast<int *>(alloc(4 * ((size_t)nc + 1)));
  C.dinv = static_cast<double *>(alloc(8 * (size_t)std::max(nc, 1)));
  int *cc = static_cast<int *>(tmp(4 * ((size_t)nc + 1)));
  int *tcol = static_cast<int *>(tmp(4 * (size_t)std::max(nc, 1) * kRapCap));
  double *tval = static_cast<double *>(tmp(8 * (size_t)std::max(nc, 1) * kRapCap));
  const int gc = rap_blocks(nc, kRapWarps);
  k_rs_rap<kRapHash, kRapWarps><<<gc, 32 * kRapWarps, 0, st>>>(nc, L.rrow, L.rcol, L.rval, L.rowptr, L.col, L.val,
                                                               L.prow, L.pcol, L.pval, cc, tcol, tval, C.dinv,
                                                               s->status);
  note_launches(1);
  scan_exclusive(s->ctx, cc, C.rowptr, nc, false);
  C.d_sys_start = static_cast<int *>(alloc(4 * ((size_t)ns + 1)));
  k_rs_coarse_starts<<<grid_for(ns + 1, TB), TB, 0, st>>>(ns, L.d_sys_start, cidx, C.d_sys_start);
  note_launches(1);
  VAG_CHECK_LAUNCH();
  // one wait for the coarse nonzeros, the status and the row starts
  int *starts = static_cast<int *>(ctx_stage(s->ctx, 4 * ((size_t)ns + 1)));
  VAG_CUDA(cudaMemcpyAsync(&pin[0], C.rowptr + nc, sizeof(int), cudaMemcpyDeviceToHost, st));
  VAG_CUDA(cudaMemcpyAsync(&pin[1], s->status, sizeof(int), cudaMemcpyDeviceToHost, st));
  VAG_CUDA(cudaMemcpyAsync(starts, C.d_sys_start, 4 * ((size_t)ns + 1), cudaMemcpyDeviceToHost, st));
  VAG_CUDA(cudaStreamSynchronize(st));
  C.sys_start.assign(starts, starts + ns + 1);
  C.nnz = pin[0];
  {
    const int stv = pin[1];
    if (stv & ST_ROW_OVERFLOW) fail(VAG_EMESH, "AMG: a coarse row couples too many coarse rows");
    if (stv & ST_NONPOSITIVE)
      fail(VAG_EINVAL, "AMG: a fine row has no usable coarse couplings or a coarse diagonal is not positive");
  }
  C.col = static_cast<int *>(alloc(4 * (size_t)std::max<int64_t>(C.nnz, 1)));
  C.val = static_cast<double *>(alloc(8 * (size_t)std::max<int64_t>(C.nnz, 1)));
  k_rs_compact<kRapCap><<<grid_for(nc, TB / 32), TB, 0, st>>>(nc, tcol, tval, C.rowptr, C.col, C.val);
  note_launches(1);
  trace_mark(st, "  classical: Galerkin R A P");
  VAG_CHECK_LAUNCH();
}

}  // namespace vag
