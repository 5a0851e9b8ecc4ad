// Build of the sliced layout of a large matrix (spmv_slice.cuh), on the device:
// a warp per window of 64 rows sorts them and cuts the slices, scans place them,
// and a warp per window copies values and columns.
#include <algorithm>
#include <cstdint>

#include "context.h"

namespace pdhg {

namespace {

constexpr int kWarps = 8;
static_assert(kSliceRows == 64, "a lane takes two rows of a window");

struct Cut {  // of one window: rows of each class, and where its slices start
  int n32, n8, n1, lg1;  // rows with 32, 8 and 2^lg1 lanes
  __device__ __forceinline__ int s8() const { return (n8 + 3) / 4; }
  __device__ __forceinline__ int slices() const { return n32 + s8() + ((n1 << lg1) + 31) / 32; }
  // lanes per row (log2), first position and rows of slice s
  __device__ __forceinline__ void slice(int s, int& lg, int& p0, int& rows) const {
    if (s < n32)
      lg = 5, p0 = s, rows = 1;
    else if (s < n32 + s8())
      lg = 3, p0 = n32 + 4 * (s - n32), rows = min(4, n32 + n8 - p0);
    else
      lg = lg1, p0 = n32 + n8 + (32 >> lg1) * (s - n32 - s8()), rows = min(32 >> lg1, n32 + n8 + n1 - p0);
  }
};

// The window's lengths sorted: key[p] the length at position p, at[p] its row.
// A warp works on its own window; ends warp-synchronised.
__device__ __forceinline__ Cut sort_window(int nrows, int q, const int32_t* __restrict__ rp, int lg1,
                                           int* key, uint8_t* at) {
  const int lane = threadIdx.x & 31, row0 = q * kSliceRows, nr = min(kSliceRows, nrows - row0);
  int len[2];
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int i = lane + 32 * h;
    len[h] = i < nr ? rp[row0 + i + 1] - rp[row0 + i] : -1;
  }
  int rank[2] = {0, 0};
#pragma unroll
  for (int h = 0; h < 2; ++h)
    for (int l = 0; l < 32; ++l) {
      const int other = __shfl_sync(0xffffffffu, len[h], l), j = l + 32 * h;
#pragma unroll
      for (int k = 0; k < 2; ++k)
        rank[k] += other > len[k] || (other == len[k] && j < lane + 32 * k);
    }
  int n32 = 0, n8 = 0;
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    key[rank[h]] = len[h];
    at[rank[h]] = (uint8_t)(lane + 32 * h);
    n32 += __popc(__ballot_sync(0xffffffffu, len[h] > kSliceMid));
    n8 += __popc(__ballot_sync(0xffffffffu, len[h] > kSliceShort << lg1 && len[h] <= kSliceMid));
  }
  __syncwarp();
  return Cut{n32, n8, nr - n32 - n8, lg1};
}

__global__ void __launch_bounds__(kWarps * 32)
    k_sl_count(int nrows, int nwin, int lg1, const int32_t* __restrict__ rp, uint8_t* ord, int32_t* count,
               int32_t* elems, unsigned long long* padded) {
  __shared__ int key[kWarps][kSliceRows];
  __shared__ uint8_t at[kWarps][kSliceRows];
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31, q = blockIdx.x * kWarps + w;
  if (q >= nwin) return;  // warp-uniform
  const Cut c = sort_window(nrows, q, rp, lg1, key[w], at[w]);
  for (int p = lane; p < c.n32 + c.n8 + c.n1; p += 32) ord[(size_t)q * kSliceRows + p] = at[w][p];
  int e = 0;
  for (int s = lane; s < c.slices(); s += 32) {
    int lg, p0, rows;
    c.slice(s, lg, p0, rows);
    e += (key[w][p0] + (1 << lg) - 1) >> lg;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) e += __shfl_xor_sync(0xffffffffu, e, o);
  if (lane == 0) {
    count[q] = c.slices();
    elems[q] = e * 32;
    atomicAdd(padded, (unsigned long long)(e * 32));
  }
}

__global__ void __launch_bounds__(kWarps * 32)
    k_sl_fill(int nrows, int ncols, int nwin, int lg1, const int32_t* __restrict__ rp, const int32_t* __restrict__ col,
              const double* __restrict__ val, const int32_t* __restrict__ slice0,
              const int32_t* __restrict__ elem0, int4* out, int32_t* col_s, double* v64) {
  __shared__ int key[kWarps][kSliceRows];
  __shared__ uint8_t at[kWarps][kSliceRows];
  const int wi = threadIdx.x >> 5, lane = threadIdx.x & 31, q = blockIdx.x * kWarps + wi;
  if (q >= nwin) return;
  const Cut c = sort_window(nrows, q, rp, lg1, key[wi], at[wi]);
  int64_t off = elem0[q];
  for (int s = 0; s < c.slices(); ++s) {
    int lg, p0, rows;
    c.slice(s, lg, p0, rows);
    const int G = 1 << lg, row = lane >> lg, gl = lane & (G - 1), w = (key[wi][p0] + G - 1) >> lg;
    if (lane == 0)
      out[slice0[q] + s] = make_int4((int)off, w | (lg << 8) | (rows << 12), q * kSliceRows + p0,
                                     q * kSliceRows);
    int b = 0, len = 0;
    if (row < rows) {
      b = rp[q * kSliceRows + at[wi][p0 + row]];
      len = key[wi][p0 + row];
    }
#pragma unroll 4
    for (int k = 0; k < w; ++k) {
      const int j = k * G + gl;
      const bool in = j < len;
      col_s[off + k * 32 + lane] = in ? col[b + j] : ncols;
      v64[off + k * 32 + lane] = in ? val[b + j] : 0.0;
    }
    off += 32 * w;
  }
}

}  // namespace

// log2 of the lanes of a short row: 1, or 2 or 4 lanes where that leaves the SMs
// fewer than kSliceWarps warps
static int short_lanes(const pdhg_ctx* ctx, bool on_a) {
  const int64_t rows = on_a ? ctx->m : ctx->n;
  int lg = 0;
  while (lg < 2 && (rows << lg) < (int64_t)32 * kSliceWarps * ctx->nsm && ctx->nnz >= rows << (lg + 2)) ++lg;
  return lg;
}

// The rule for slices in place of tiles: from 2^16 nonzeros on where the LP is
// not solved on chip and no tile capacity is forced, and where the chain of steps
// of a row that has a warp to itself is short beside the whole.  A step of a lone warp takes about
// 0.2 us and a million nonzeros 3.7 us in slices and 7 in tiles.  Float64 A~ of
// transportation LPs (rows as long as the other side), tiles / slices, us:
// 2000 x 2000 (62 steps, 8 million) 61 / 42, 1200 x 1900 39 / 22, 700 x 900 13.9 /
// 10.9, 400 x 400 (13 steps) 7.1 / 5.8; 301 x 707 (22 steps, 0.4 million) 7.7 /
// 7.6; and left to the tiles 1000 x 300 (31 steps, 0.6 million) 7.9 / 11.1,
// 200 x 2000 10.8 / 16.1, 1900 x 40 6.4 / 13.5.
bool slices_pay(const pdhg_ctx* ctx, bool on_a) {
  if (ctx->batch || ctx->resident || ctx->opt.tile_nnz != 0 || ctx->nnz < (1 << 16)) return false;
  const int longest = on_a ? ctx->longest_a : ctx->longest_t, steps = (longest + 31) / 32;
  return longest <= kSliceMid || (steps <= kSliceMaxSteps && steps <= 14 + (int)(ctx->nnz >> 16));
}

// The sliced schedule of A~ (on_a) or A~^T with its float64 values; no slice
// has more than kSliceMaxSteps steps (slices_pay).
// d->view.e stays 0, and the matrix is left to the tiles, where rows of very
// different lengths share windows (more padding than nonzeros) or where the
// copy would take more than a quarter of the memory that is left.
static pdhg_status make_slices(pdhg_ctx* ctx, bool on_a, DevSched* d) {
  *d = DevSched{};
  const int nrows = on_a ? ctx->m : ctx->n, ncols = on_a ? ctx->n : ctx->m;
  const int32_t *rp = on_a ? ctx->a_rp : ctx->t_rp, *col = on_a ? ctx->a_col : ctx->t_col;
  const double* val = on_a ? ctx->a_val64 : ctx->t_val64;
  cudaStream_t s = ctx->stream;
  const int nw = (nrows + kSliceRows - 1) / kSliceRows, grid = (nw + kWarps - 1) / kWarps;
  const int lg1 = short_lanes(ctx, on_a);
  int4* slices = nullptr;
  uint8_t* ord = nullptr;
  int32_t *elems = nullptr, *elem0 = nullptr, *count = nullptr, *slice0 = nullptr, *tmp = nullptr,
          *scol = nullptr;
  unsigned long long *padded = nullptr, total = 0;
  double* v64 = nullptr;
  CKS(dalloc(ctx, &ord, (size_t)nw * kSliceRows));
  CKS(dalloc(ctx, &count, (size_t)nw));
  CKS(dalloc(ctx, &slice0, (size_t)nw + 1));
  CKS(dalloc(ctx, &elems, (size_t)nw));
  CKS(dalloc(ctx, &elem0, (size_t)nw + 1));
  CKS(dalloc(ctx, &tmp, (size_t)nw / 1024 + 8));
  CKS(dalloc(ctx, &padded, 1));
  CK(cudaMemsetAsync(padded, 0, sizeof(*padded), s));
  k_sl_count<<<grid, kWarps * 32, 0, s>>>(nrows, nw, lg1, rp, ord, count, elems, padded);
  launch_scan(elems, elem0, nw, tmp, s);
  launch_scan(count, slice0, nw, tmp, s);
  ctx->launches += 7;
  int32_t nslices = 0;
  CK(cudaMemcpyAsync(&nslices, slice0 + nw, sizeof(nslices), cudaMemcpyDeviceToHost, s));
  CK(cudaMemcpyAsync(&total, padded, sizeof(total), cudaMemcpyDeviceToHost, s));
  CK(cudaStreamSynchronize(s));
  if (total > (unsigned long long)ctx->nnz * 2 || total > (unsigned long long)INT32_MAX) return PDHG_OK;
  const size_t bytes = (size_t)total * 12;
  size_t left = 0, all = 0;
  if (bytes > (size_t(1) << 28)) {
    CK(cudaMemGetInfo(&left, &all));
    if (bytes > left / 4) return PDHG_OK;
  }
  CKS(dalloc(ctx, &slices, (size_t)nslices));
  CKS(dalloc(ctx, &scol, (size_t)total));
  CKS(dalloc(ctx, &v64, (size_t)total));
  k_sl_fill<<<grid, kWarps * 32, 0, s>>>(nrows, ncols, nw, lg1, rp, col, val, slice0, elem0, slices, scol, v64);
  ctx->launches += 1;
  CK(cudaGetLastError());
  SchedView& V = d->view;
  V.ntiles = (nslices + kBlock / 32 - 1) / (kBlock / 32);
  V.tile_nnz = 32 * kSliceMaxSteps;
  V.max_rows = kSliceRows;
  V.e = kSliced;
  V.nslices = nslices;
  V.slices = slices;
  V.slice_ord = ord;
  V.slice_col = scol;
  V.slice_val = v64;
  return PDHG_OK;
}

pdhg_status build_slices(pdhg_ctx* ctx, bool on_a, DevSched* d) {
  return if_room(ctx, [&] { return make_slices(ctx, on_a, d); }, [&] { *d = DevSched{}; });
}

}  // namespace pdhg
