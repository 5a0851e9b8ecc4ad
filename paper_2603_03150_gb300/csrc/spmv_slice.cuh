// Sliced SpMV core: the row-sorted counterpart of run_tiles (spmv_tile.cuh) for
// large matrices whose longest row is short beside the whole (slices_pay in
// slices.cu), with the same epilogues.
//
// Windows of kSliceRows rows are sorted by length (longest first, equal lengths
// in row order); rows of up to kSliceShort nonzeros go 32 to a slice (a lane
// each; 2 or 4 on small matrices), those of up to kSliceMid 4 to a slice (8 lanes
// each), longer ones one to a slice.  Step k of a slice is 32 consecutive values
// and columns; past a row's end the value is 0 and the column the one behind the
// last, where every gathered vector holds a 0 (a column that the row does not hold
// could hold an infinity or a NaN, which a value of 0 would carry into the sum).  A warp takes a slice: a row costs one multiply-add per nonzero
// (and the additions of a shuffle sum in the longer classes) where run_tiles adds
// a segmented scan of 5 additions for 8 nonzeros, and there is no block barrier
// and no staging: the lane that holds a row's sum runs its epilogue, whose
// operands it has loaded before the sum.
//
// What bounds it is latency (ncu, A~^T of the power-law LP, float64: long
// scoreboard 31 of 39 cycles per issued instruction, float64 pipe 30%).  Per
// half-step kernel, tiles of 8 nonzeros per thread against slices, float64: A~^T
// (5 nonzeros a row) of the planted LP 100,000 x 250,000 16.5 -> 9.7 us, its A~
// (12.5) 15.8 -> 11.4, A~^T of the power-law LP 43.8 -> 35.4, A~^T of the
// transportation LP 2000 x 2000 (2) 77 -> 52.  Windows: the lanes' accesses stay within
// a window, so wider ones sort better but scatter more: A~^T of the power-law
// LP 36.6 / 39.2 / 42.2 us at 64 / 128 / 256 rows.  Cutting longer rows into
// chunks did not pay: power-law A~ (rows up to 20,000) 49 us against the tiles'
// 43.5.
#pragma once
#include "spmv_tile.cuh"

namespace pdhg {

__host__ __device__ constexpr int slice_steps(int w) { return w & 0xff; }
__host__ __device__ constexpr int slice_lg(int w) { return (w >> 8) & 15; }
__host__ __device__ constexpr int slice_nrows(int w) { return (w >> 12) & 63; }

// Sums of a slice: lane l gets the row l >> lg.  Four steps at a time with the
// next four's values and columns in flight; the last w mod 4 are loaded and
// gathered first and added last, in a loop of their own (a float64 operation
// whose predicate is off still takes its slot of the pipe).
template <typename T, int NV, class Gv>
__device__ __forceinline__ void slice_dot(const T* __restrict__ val, const int32_t* __restrict__ col,
                                          int w, int lg, const Gv& g, uint64_t pol, T (&acc)[NV]) {
  const int full = w & ~3;
  T a[4], ta[3], tg[3][NV];
  int j[4];
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    a[e] = T(0);
    j[e] = 0;
    if (full) {
      a[e] = ld_stream(val + e * 32, pol);
      j[e] = ld_stream(col + e * 32, pol);
    }
  }
#pragma unroll
  for (int e = 0; e < 3; ++e) {
    ta[e] = T(0);
#pragma unroll
    for (int v = 0; v < NV; ++v) tg[e][v] = T(0);
    if (full + e < w) {
      ta[e] = ld_stream(val + (full + e) * 32, pol);
      g.load(ld_stream(col + (full + e) * 32, pol), tg[e]);
    }
  }
#pragma unroll
  for (int v = 0; v < NV; ++v) acc[v] = T(0);
#pragma unroll 1
  for (int k = 0; k < full; k += 4) {
    T gv[4][NV], ca[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      ca[e] = a[e];
      g.load(j[e], gv[e]);
    }
    if (k + 4 < full) {
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        a[e] = ld_stream(val + (k + 4 + e) * 32, pol);
        j[e] = ld_stream(col + (k + 4 + e) * 32, pol);
      }
    }
#pragma unroll
    for (int e = 0; e < 4; ++e)
#pragma unroll
      for (int v = 0; v < NV; ++v) acc[v] = fmadd(ca[e], gv[e][v], acc[v]);
  }
#pragma unroll 1
  for (int e = full; e < w; ++e) {
#pragma unroll
    for (int v = 0; v < NV; ++v) acc[v] = fmadd(ta[0], tg[0][v], acc[v]);
    ta[0] = ta[1], ta[1] = ta[2];
#pragma unroll
    for (int v = 0; v < NV; ++v) tg[0][v] = tg[1][v], tg[1][v] = tg[2][v];
  }
  if (lg) {  // warp-uniform
#pragma unroll 1
    for (int o = 1 << (lg - 1); o > 0; o >>= 1)
#pragma unroll
      for (int v = 0; v < NV; ++v) acc[v] += __shfl_xor_sync(0xffffffffu, acc[v], o);
  }
}

// An epilogue with load(r) and apply(r, in, s) has its row's operands loaded
// before the row's sum is known, so the two latencies overlap (A~ of the planted
// LP above 15.8 -> 11.4 us).
struct NoOperands {};
template <class Epi>
__device__ __forceinline__ auto epi_operands(const Epi& e, int r, int) -> decltype(e.load(r)) {
  return e.load(r);
}
template <class Epi>
__device__ __forceinline__ NoOperands epi_operands(const Epi&, int, long) {
  return {};
}
template <typename T, int NV, class Epi, class In>
__device__ __forceinline__ void epi_apply(Epi& e, int r, const In& in, const T (&s)[NV]) {
  if constexpr (std::is_same<In, NoOperands>::value)
    e.row(r, s, -1);
  else if constexpr (NV == 1)
    e.apply(r, in, s[0]);
  else
    e.apply(r, in, s);
}

template <typename T, int NV, int BLOCK, class Epi, class Gv>
__device__ __forceinline__ void run_slices(const SchedView& S, const Gv& g, Epi& epi) {
  constexpr int NW = BLOCK / 32;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint64_t pol = stream_policy();
  const T* sval = reinterpret_cast<const T*>(S.slice_val);
  const int step = gridDim.x * NW;
  int s = blockIdx.x * NW + warp;
  int4 d = s < S.nslices ? __ldg(S.slices + s) : make_int4(0, 0, 0, 0);
  while (s < S.nslices) {
    const int lg = slice_lg(d.y), row = lane >> lg, w = slice_steps(d.y);
    const bool mine = (lane & ((1 << lg) - 1)) == 0 && row < slice_nrows(d.y);
    // lanes without a row read the operands of the window's first
    const int r = d.w + (mine ? __ldg(S.slice_ord + d.z + row) : 0);
    const size_t at = (size_t)d.x + lane;
    s += step;
    if (s < S.nslices) d = __ldg(S.slices + s);
    const auto in = epi_operands(epi, r, 0);
    T acc[NV];
    slice_dot<T, NV>(sval + at, S.slice_col + at, w, lg, g, pol, acc);
    if (mine) epi_apply(epi, r, in, acc);
  }
}

// Schedule variant V: V = kSliced the slices above, V > 0 segmented tiles with
// E = V nonzeros per thread, V < 0 vector tiles with G = -V lanes per row.
template <typename T, int NV, int BLOCK, int V, class Epi, class Gv>
__device__ __forceinline__ void run_sched(const SchedView& S, const int32_t* __restrict__ row_ptr,
                                          const int32_t* __restrict__ col,
                                          const T* __restrict__ val, const Gv& g,
                                          Epi& epi, unsigned char* smem) {
  if constexpr (V == kSliced)
    run_slices<T, NV, BLOCK>(S, g, epi);
  else if constexpr (V > 0)
    run_tiles<T, NV, BLOCK, V>(S, row_ptr, col, val, g, epi, smem);
  else
    run_tiles_vec<T, NV, BLOCK, -V>(S, row_ptr, col, val, g, epi, smem);
}

}  // namespace pdhg
