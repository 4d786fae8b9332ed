// Sliced-ELL copy (slices of 32 consecutive rows, column-major inside a
// slice) of the eliminated system, for thread-per-row SpMV: the 32 threads of
// a warp read entry k of their 32 rows as one contiguous 256-byte (FP64) or
// 128-byte (FP32) segment, and a row costs exactly one FMA per stored entry
// (no cross-lane reduction -- on GB300 the FP64 pipe, not HBM, limits a
// lane-split CSR SpMV).  Entries of a row keep their CSR order, so a row sum
// is the same sequence of FMAs whatever the slice layout.
#include <climits>

#include "vag_internal.cuh"

namespace vag {
namespace {

constexpr int TB = 256;

__global__ void k_slice_width(int n, int n_slices, const int *__restrict__ rowptr, int *__restrict__ width) {
  const int sl = blockIdx.x * blockDim.x + threadIdx.x;
  if (sl >= n_slices) return;
  int w = 0;
  const int r1 = min(n, (sl + 1) * 32);
  for (int r = sl * 32; r < r1; ++r) w = max(w, rowptr[r + 1] - rowptr[r]);
  width[sl] = 32 * w;
}

__global__ void k_sell_cols(int n, const int *__restrict__ rowptr, const int *__restrict__ col,
                            const int *__restrict__ slice_ptr, int *__restrict__ scol) {
  const int row = blockIdx.x * blockDim.x + threadIdx.x;
  if (row >= n) return;
  const int b = rowptr[row], e = rowptr[row + 1];
  const int base = slice_ptr[row >> 5] + (row & 31);
  for (int k = 0; k < e - b; ++k) scol[base + 32 * k] = col[b + k];
}

// padding slots point at the row itself (their values are 0)
__global__ void k_sell_pad(int n, const int *__restrict__ rowptr, const int *__restrict__ slice_ptr,
                           int *__restrict__ scol) {
  const int row = blockIdx.x * blockDim.x + threadIdx.x;
  if (row >= ((n + 31) / 32) * 32) return;
  const int sl = row >> 5;
  const int w = (slice_ptr[sl + 1] - slice_ptr[sl]) / 32;
  const int len = row < n ? rowptr[row + 1] - rowptr[row] : 0;
  const int base = slice_ptr[sl] + (row & 31);
  for (int k = len; k < w; ++k) scol[base + 32 * k] = row < n ? row : 0;
}

// One warp per slice: the slice's smallest column and the 16-bit offsets from
// it, or -1 where they do not fit (the columns then stay 32-bit).
__global__ void __launch_bounds__(TB) k_sell_pack(int n, int n_slices, const int *__restrict__ slice_ptr,
                                                  const int *__restrict__ scol, unsigned short *__restrict__ c16,
                                                  int *__restrict__ sbase) {
  const int sl = blockIdx.x * (TB / 32) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (sl >= n_slices) return;   // whole warps
  const int b = slice_ptr[sl], e = slice_ptr[sl + 1];
  const bool mine = sl * 32 + lane < n;   // past the last row the columns are 0
  int lo = INT_MAX, hi = -1;
  for (int p = b + lane; p < e; p += 32) {
    const int c = scol[p];
    if (mine) {
      lo = min(lo, c);
      hi = max(hi, c);
    }
  }
  lo = __reduce_min_sync(0xffffffffu, lo);
  hi = __reduce_max_sync(0xffffffffu, hi);
  const bool fits = hi >= 0 && hi - lo < 65536;
  if (lane == 0) sbase[sl] = fits ? lo : -1;
  if (!fits) return;
  for (int p = b + lane; p < e; p += 32) c16[p] = mine ? (unsigned short)(scol[p] - lo) : (unsigned short)0;
}

template <class T>
__device__ __forceinline__ T to_store(double v) { return (T)v; }
template <>
__device__ __forceinline__ __half to_store<__half>(double v) { return __double2half(v); }

template <class T>
__global__ void k_sell_vals(int n, const int *__restrict__ rowptr, const double *__restrict__ val,
                            const double *__restrict__ scale, const int *__restrict__ col,
                            const int *__restrict__ slice_ptr, T *__restrict__ sval) {
  const int row = blockIdx.x * blockDim.x + threadIdx.x;
  if (row >= n) return;
  const int b = rowptr[row], e = rowptr[row + 1];
  const int base = slice_ptr[row >> 5] + (row & 31);
  const double sr = scale ? scale[row] : 1.0;
  for (int k = 0; k < e - b; ++k) {
    const double v = scale ? sr * val[b + k] * scale[col[b + k]] : val[b + k];
    sval[base + 32 * k] = to_store<T>(v);
  }
  // padding up to the slice width: value 0 (its column is the row itself)
  const int w = (slice_ptr[(row >> 5) + 1] - slice_ptr[row >> 5]) >> 5;
  for (int k = e - b; k < w; ++k) sval[base + 32 * k] = to_store<T>(0.0);
}

}  // namespace

void sell_slices(System *s) {
  cudaStream_t st = s->ctx->stream;
  s->n_slices = (s->n_rows + 31) / 32;
  s->slice_ptr = sys_alloc<int>(s, (size_t)s->n_slices + 1);
  Scratch scratch(s->ctx);
  int *width = scratch.get<int>((size_t)s->n_slices + 1);
  k_slice_width<<<grid_for(s->n_slices, TB), TB, 0, st>>>(s->n_rows, s->n_slices, s->rowptr, width);
  note_launches(1);
  VAG_CHECK_LAUNCH();
  scan_exclusive(s->ctx, width, s->slice_ptr, s->n_slices, false);
}

void build_sell(System *s, int64_t total) {
  cudaStream_t st = s->ctx->stream;
  const int n = s->n_rows;
  s->sell_nnz = total;
  s->scol = sys_alloc<int>(s, (size_t)std::max<int64_t>(total, 1));
  s->sval = sys_alloc<double>(s, (size_t)std::max<int64_t>(total, 1));
  if (n > 0) {
    k_sell_cols<<<grid_for(n, TB), TB, 0, st>>>(n, s->rowptr, s->col, s->slice_ptr, s->scol);
    k_sell_pad<<<grid_for((int64_t)s->n_slices * 32, TB), TB, 0, st>>>(n, s->rowptr, s->slice_ptr, s->scol);
    note_launches(2);
    // (a context with a budget keeps to the arrays that the budget was set for)
    if ((size_t)total * 12 > kStreamBytes && !s->ctx->budget) {
      s->scol16 = sys_alloc<unsigned short>(s, (size_t)total);
      s->sbase = sys_alloc<int>(s, (size_t)s->n_slices);
      k_sell_pack<<<grid_for(s->n_slices, TB / 32), TB, 0, st>>>(n, s->n_slices, s->slice_ptr, s->scol, s->scol16,
                                                                 s->sbase);
      note_launches(1);
    }
    VAG_CHECK_LAUNCH();
  }
}

void sell_values(System *s) {
  cudaStream_t st = s->ctx->stream;
  k_sell_vals<double><<<grid_for(s->n_rows, TB), TB, 0, st>>>(s->n_rows, s->rowptr, s->val, nullptr, s->col,
                                                               s->slice_ptr, s->sval);
  note_launches(1);
  VAG_CHECK_LAUNCH();
}

// FP32 copy of D^{-1/2} A D^{-1/2} (scale = D^{-1/2}, FP64) for the inner
// solve of the mixed-precision path.
void sell_values_scaled_f32(System *s, const double *scale, float *out) {
  cudaStream_t st = s->ctx->stream;
  k_sell_vals<float><<<grid_for(s->n_rows, TB), TB, 0, st>>>(s->n_rows, s->rowptr, s->val, scale, s->col,
                                                              s->slice_ptr, out);
  note_launches(1);
  VAG_CHECK_LAUNCH();
}

void sell_values_f32(System *s, float *out) { sell_values_scaled_f32(s, nullptr, out); }

// FP16 copy of D^{-1/2} A D^{-1/2} (scale = D^{-1/2}, FP64): unit diagonal,
// off-diagonal entries in [-1, 1], so FP16 keeps about three digits of each.
void sell_values_scaled_f16(System *s, const double *scale, __half *out) {
  cudaStream_t st = s->ctx->stream;
  k_sell_vals<__half><<<grid_for(s->n_rows, TB), TB, 0, st>>>(s->n_rows, s->rowptr, s->val, scale, s->col,
                                                               s->slice_ptr, out);
  note_launches(1);
  VAG_CHECK_LAUNCH();
}

}  // namespace vag
