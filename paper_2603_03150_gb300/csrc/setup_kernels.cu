// Set-up kernels: CSR validation, stable transpose, diagonal scaling (Ruiz and
// Pock-Chambolle statistics), scaled copies, reductions and power iteration.
#include <algorithm>
#include <math.h>

#include "dispatch.cuh"
#include "kernels.h"
#include "spmv_slice.cuh"

namespace pdhg {

static int grid_cap(int64_t work, int per_block = 256, int cap = 8192) {
  int64_t g = (work + per_block - 1) / per_block;
  if (g > cap) g = cap;
  return g < 1 ? 1 : (int)g;
}

// ---------------------------------------------------------------------------
// validation: flags |= 1 column out of range, 2 columns not strictly
// increasing in a row, 4 non-finite value, 8 non-finite b, 16 non-finite c
// ---------------------------------------------------------------------------
__global__ void k_validate(int m, int n, const int32_t* rp, const int32_t* col, const double* val,
                           const double* b, const double* c, int32_t* flags) {
  int f = 0;
  each_nonzero(m, rp, [&](int k, int i) {
    const int cj = col[k];
    if (cj < 0 || cj >= n) f |= 1;
    if (k > rp[i] && col[k - 1] >= cj) f |= 2;
    if (!isfinite(val[k])) f |= 4;
  });
  const int tid = blockIdx.x * blockDim.x + threadIdx.x, nt = gridDim.x * blockDim.x;
  for (int i = tid; i < m; i += nt)
    if (!isfinite(b[i])) f |= 8;
  for (int j = tid; j < n; j += nt)
    if (!isfinite(c[j])) f |= 16;
  if (f) atomicOr(flags, f);
}

void launch_validate(int m, int n, int64_t nnz, const int32_t* rp, const int32_t* col, const double* val,
                     const double* b, const double* c, int32_t* flags, cudaStream_t s) {
  k_validate<<<grid_cap(std::max<int64_t>({nnz / 8, m, n})), 256, 0, s>>>(m, n, rp, col, val, b, c, flags);
}

// ---------------------------------------------------------------------------
// transpose: column histogram, exclusive scan, scatter, per-column sort
// ---------------------------------------------------------------------------
__global__ void k_col_hist(int64_t nnz, const int32_t* col, int32_t* cnt) {
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < nnz;
       k += (int64_t)gridDim.x * blockDim.x)
    atomicAdd(cnt + col[k], 1);
}
void launch_col_hist(int64_t nnz, const int32_t* col, int32_t* cnt, cudaStream_t s) {
  k_col_hist<<<grid_cap(nnz), 256, 0, s>>>(nnz, col, cnt);
}

constexpr int kScanT = 256, kScanPer = 4, kScanTile = kScanT * kScanPer;

__device__ __forceinline__ int warp_incl_scan(int v) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int t = __shfl_up_sync(0xffffffffu, v, o);
    if (lane >= o) v += t;
  }
  return v;
}

// exclusive scan of one 1024-element tile; tile total -> tops[blockIdx]
__global__ void k_scan_tile(const int32_t* in, int32_t* out, int len, int32_t* tops) {
  __shared__ int wsum[kScanT / 32];
  const int base = blockIdx.x * kScanTile + threadIdx.x * kScanPer;
  int v[kScanPer], s = 0;
#pragma unroll
  for (int e = 0; e < kScanPer; ++e) {
    v[e] = (base + e < len) ? in[base + e] : 0;
    s += v[e];
  }
  const int incl = warp_incl_scan(s);
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  if (lane == 31) wsum[w] = incl;
  __syncthreads();
  if (w == 0) {
    int x = (lane < kScanT / 32) ? wsum[lane] : 0;
    x = warp_incl_scan(x);
    if (lane < kScanT / 32) wsum[lane] = x;
  }
  __syncthreads();
  int run = incl - s + (w > 0 ? wsum[w - 1] : 0);
#pragma unroll
  for (int e = 0; e < kScanPer; ++e) {
    if (base + e < len) out[base + e] = run;
    run += v[e];
  }
  if (threadIdx.x == kScanT - 1) tops[blockIdx.x] = run;
}

// exclusive scan of the tile totals in one block (sequential over chunks)
__global__ void k_scan_tops(int32_t* tops, int ntiles, int32_t* total_out) {
  __shared__ int carry;
  if (threadIdx.x == 0) carry = 0;
  __syncthreads();
  for (int base = 0; base < ntiles; base += blockDim.x) {
    const int i = base + threadIdx.x;
    const int v = (i < ntiles) ? tops[i] : 0;
    // block-wide inclusive scan of blockDim.x (= 1024) values
    __shared__ int ws[32];
    const int incl = warp_incl_scan(v);
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if (lane == 31) ws[w] = incl;
    __syncthreads();
    if (w == 0) {
      int x = ws[lane];
      x = warp_incl_scan(x);
      ws[lane] = x;
    }
    __syncthreads();
    const int excl = incl - v + (w > 0 ? ws[w - 1] : 0) + carry;
    if (i < ntiles) tops[i] = excl;
    __syncthreads();
    if (threadIdx.x == blockDim.x - 1) carry = excl + v;
    __syncthreads();
  }
  if (threadIdx.x == 0) *total_out = carry;
}

__global__ void k_scan_add(int32_t* out, int len, const int32_t* tops) {
  const int i = blockIdx.x * kScanTile + threadIdx.x;
  const int add = tops[blockIdx.x];
#pragma unroll
  for (int e = 0; e < kScanPer; ++e) {
    const int k = i + e * kScanT;
    if (k < len) out[k] += add;
  }
}

void launch_scan(const int32_t* cnt, int32_t* out, int len, int32_t* tmp, cudaStream_t s) {
  const int ntiles = (len + kScanTile - 1) / kScanTile;
  if (ntiles == 0) {
    cudaMemsetAsync(out, 0, sizeof(int32_t), s);
    return;
  }
  k_scan_tile<<<ntiles, kScanT, 0, s>>>(cnt, out, len, tmp);
  k_scan_tops<<<1, 1024, 0, s>>>(tmp, ntiles, out + len);
  k_scan_add<<<ntiles, kScanT, 0, s>>>(out, len, tmp);
}

__global__ void k_scatter(int m, const int32_t* rp, const int32_t* col, const double* val,
                          int32_t* cursor, int32_t* col_t, double* val_t) {
  each_nonzero(m, rp, [&](int k, int i) {
    const int pos = atomicAdd(cursor + col[k], 1);
    col_t[pos] = i;
    val_t[pos] = val[k];
  });
}
void launch_scatter(int m, int64_t nnz, const int32_t* rp, const int32_t* col, const double* val,
                    int32_t* cursor, int32_t* col_t, double* val_t, cudaStream_t s) {
  k_scatter<<<grid_cap(nnz / 8), 256, 0, s>>>(m, rp, col, val, cursor, col_t, val_t);
}

// segments of <= 32 entries: one thread, insertion sort in place
__global__ void k_segsort_small(int nseg, const int32_t* seg, int32_t* keys, double* vals) {
  for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < nseg; j += gridDim.x * blockDim.x) {
    const int s = seg[j], e = seg[j + 1];
    if (e - s > 32 || e - s < 2) continue;
    for (int a = s + 1; a < e; ++a) {
      const int kk = keys[a];
      const double vv = vals[a];
      int b = a - 1;
      while (b >= s && keys[b] > kk) {
        keys[b + 1] = keys[b];
        vals[b + 1] = vals[b];
        --b;
      }
      keys[b + 1] = kk;
      vals[b + 1] = vv;
    }
  }
}

constexpr int kBitonicMax = 2048;

// longer segments: one block each; bitonic sort in shared memory up to 2048
// entries, else rank by counting (keys within a segment are distinct rows)
__global__ void __launch_bounds__(1024) k_segsort_long(const int32_t* seg, int32_t* keys, double* vals,
                                                       const int32_t* ids, int32_t* tmp_k,
                                                       double* tmp_v) {
  __shared__ int sk[kBitonicMax];
  __shared__ double sv[kBitonicMax];
  const int j = ids[blockIdx.x];
  const int s = seg[j], e = seg[j + 1], len = e - s;
  if (len <= kBitonicMax) {
    int p2 = 1;
    while (p2 < len) p2 <<= 1;
    for (int i = threadIdx.x; i < p2; i += blockDim.x) {
      sk[i] = (i < len) ? keys[s + i] : 0x7fffffff;
      sv[i] = (i < len) ? vals[s + i] : 0.0;
    }
    __syncthreads();
    for (int size = 2; size <= p2; size <<= 1)
      for (int stride = size >> 1; stride > 0; stride >>= 1) {
        for (int i = threadIdx.x; i < p2; i += blockDim.x) {
          const int pr = i ^ stride;
          if (pr > i) {
            const bool up = (i & size) == 0;
            if ((sk[i] > sk[pr]) == up) {
              const int tk = sk[i];
              sk[i] = sk[pr];
              sk[pr] = tk;
              const double tv = sv[i];
              sv[i] = sv[pr];
              sv[pr] = tv;
            }
          }
        }
        __syncthreads();
      }
    for (int i = threadIdx.x; i < len; i += blockDim.x) {
      keys[s + i] = sk[i];
      vals[s + i] = sv[i];
    }
    return;
  }
  for (int a = threadIdx.x; a < len; a += blockDim.x) {
    const int ka = keys[s + a];
    int rank = 0;
    for (int b = 0; b < len; ++b) rank += (keys[s + b] < ka) ? 1 : 0;
    tmp_k[s + rank] = ka;
    tmp_v[s + rank] = vals[s + a];
  }
  __syncthreads();
  for (int a = threadIdx.x; a < len; a += blockDim.x) {
    keys[s + a] = tmp_k[s + a];
    vals[s + a] = tmp_v[s + a];
  }
}

void launch_segsort(int nseg, const int32_t* seg_ptr, int32_t* keys, double* vals,
                    const int32_t* long_ids, int n_long, int32_t* tmp_k, double* tmp_v,
                    cudaStream_t s) {
  k_segsort_small<<<grid_cap(nseg), 256, 0, s>>>(nseg, seg_ptr, keys, vals);
  if (n_long > 0) k_segsort_long<<<n_long, 1024, 0, s>>>(seg_ptr, keys, vals, long_ids, tmp_k, tmp_v);
}

// ---------------------------------------------------------------------------
// scaling statistics of D_self M D_other and scaled copies
// ---------------------------------------------------------------------------
// d_new[i] = d_self[i] divided by the row statistic sqrt(d_self[i] * max_j
// |M_ij| d_other[j]) (mode 0) or sqrt(d_self[i] * sum_j |M_ij| d_other[j])
// (mode 1); zero -> 1.  Bound by the float64 pipe: the products, and the root
// and quotient of each row.  G lanes take a row (G sized to the mean row
// length), a warp RPW rows at a time; their statistics are collected one to a
// lane over `passes` passes and the roots and quotients taken at once: a root in
// the one lane that holds a row's statistic costs the pipe as much as 32.
// Power-law LP: 200,000 rows of A 156 -> 78 us, 1,000,000 of A^T 108 -> 74 us,
// the division pass after each (11 us) and a launch per matrix for the rows
// longer than long_len (60 us; here the first nlong blocks, one row each) gone.
// mode 0 takes the maximum on the bit patterns of the non-negative products
// (ordered like the values), off the float64 pipe.
__device__ __forceinline__ double scaled_by_stat(double d, double acc) {
  const double r = sqrt(d * acc);
  return d / (r == 0.0 ? 1.0 : r);
}

template <int G, bool kSum>
__global__ void __launch_bounds__(256)
    k_row_stat(int nrows, const int32_t* __restrict__ rp, const int32_t* __restrict__ col,
               const double* __restrict__ val, const double* __restrict__ d_self,
               const double* __restrict__ d_other, int long_len, const int32_t* __restrict__ long_ids,
               int nlong, int passes, double* __restrict__ d_new) {
  const int lane = threadIdx.x & 31;
  if ((int)blockIdx.x < nlong) {
    __shared__ double red[8];
    const int i = long_ids[blockIdx.x], e = rp[i + 1];
    double acc = 0.0;
    long long mx = 0;
#pragma unroll 4
    for (int k = rp[i] + threadIdx.x; k < e; k += 256) {
      const double p = fabs(val[k]) * d_other[col[k]];
      if (kSum) acc += p;
      else mx = max(mx, __double_as_longlong(p));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      if (kSum) acc += __shfl_down_sync(0xffffffffu, acc, o);
      else mx = max(mx, __shfl_down_sync(0xffffffffu, mx, o));
    }
    if (lane == 0) red[threadIdx.x >> 5] = kSum ? acc : __longlong_as_double(mx);
    __syncthreads();
    if (threadIdx.x == 0) {
      double v = red[0];
      for (int w = 1; w < 8; ++w) v = kSum ? v + red[w] : fmax(v, red[w]);
      d_new[i] = scaled_by_stat(d_self[i], v);
    }
    return;
  }
  constexpr int RPW = 32 / G;  // rows per pass of a warp
  const int gw = lane / G, gl = lane & (G - 1);
  const int warp = (((int)blockIdx.x - nlong) * 256 + (int)threadIdx.x) >> 5;
  const int nw = (((int)gridDim.x - nlong) * 256) >> 5;
  const int group = passes * RPW;
  for (int base = warp * group; base < nrows; base += nw * group) {
    // the bounds of the group's rows, one to a lane
    const int i = lane < group ? base + lane : nrows;
    const int b0 = i < nrows ? rp[i] : 0, e0 = i < nrows ? rp[i + 1] : 0;
    double mine = 0.0;
#pragma unroll 4
    for (int p = 0; p < passes; ++p) {
      const int src = p * RPW + gw;
      const int b = __shfl_sync(0xffffffffu, b0, src);
      int e = __shfl_sync(0xffffffffu, e0, src);
      if (e - b > long_len) e = b;
      double acc = 0.0;
      long long mx = 0;
      for (int k = b + gl; k < e; k += G) {
        const double q = fabs(val[k]) * d_other[col[k]];
        if (kSum) acc += q;
        else mx = max(mx, __double_as_longlong(q));
      }
#pragma unroll
      for (int o = G / 2; o > 0; o >>= 1) {
        if (kSum) acc += __shfl_xor_sync(0xffffffffu, acc, o);
        else mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
      }
      const double v = __shfl_sync(0xffffffffu, kSum ? acc : __longlong_as_double(mx), (lane % RPW) * G);
      if (lane / RPW == p) mine = v;
    }
    if (i < nrows && e0 - b0 <= long_len) d_new[i] = scaled_by_stat(d_self[i], mine);
  }
}

void launch_row_stat(int nrows, const int32_t* rp, const int32_t* col, const double* val,
                     const double* d_self, const double* d_other, int mode, double* d_new,
                     const RowStatPlan& plan, cudaStream_t s) {
  // passes of a warp: all G (32 rows, full lanes in the roots) once every SM
  // has 32 warps, fewer rows a warp on smaller matrices (200 rows: 5.6 us in
  // one pass against 19 in 16)
  const int rpw = 32 / plan.lanes;
  const int passes = std::max(1, std::min(plan.lanes, nrows / (rpw * plan.nsm * 32)));
  const int g = plan.nlong + grid_cap((int64_t)nrows * 32 / (passes * rpw));
#define PDHG_ROW_STAT(G)                                                                              \
  if (mode)                                                                                           \
    k_row_stat<G, true><<<g, 256, 0, s>>>(nrows, rp, col, val, d_self, d_other, plan.long_len,       \
                                          plan.long_ids, plan.nlong, passes, d_new);                         \
  else                                                                                                \
    k_row_stat<G, false><<<g, 256, 0, s>>>(nrows, rp, col, val, d_self, d_other, plan.long_len,      \
                                           plan.long_ids, plan.nlong, passes, d_new)
  switch (plan.lanes) {
    case 4: PDHG_ROW_STAT(4); break;
    case 8: PDHG_ROW_STAT(8); break;
    case 16: PDHG_ROW_STAT(16); break;
    default: PDHG_ROW_STAT(32); break;
  }
#undef PDHG_ROW_STAT
}

__global__ void k_fill(double* d, double v, int64_t len) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < len;
       i += (int64_t)gridDim.x * blockDim.x)
    d[i] = v;
}
void launch_fill(double* d, double v, int64_t len, cudaStream_t s) {
  k_fill<<<grid_cap(len), 256, 0, s>>>(d, v, len);
}

// A~_ij = (D_r[i] A_ij) D_c[j], evaluated in that order for A and for A^T so
// both stored copies hold identical values.  For A^T rows are columns of A.
__global__ void k_scale_vals(int nrows, const int32_t* rp, const int32_t* col, const double* val,
                             const double* d_row, const double* d_col, int transposed,
                             double* out64, float* out32) {
  each_nonzero(nrows, rp, [&](int k, int i) {
    const double dr = transposed ? d_row[col[k]] : d_row[i];
    const double dc = transposed ? d_col[i] : d_col[col[k]];
    const double v = (dr * val[k]) * dc;
    out64[k] = v;
    if (out32) out32[k] = (float)v;
  });
}
void launch_scale_vals(int nrows, int64_t nnz, const int32_t* rp, const int32_t* col, const double* val,
                       const double* D_r, const double* D_c, int transposed, double* out64,
                       float* out32, cudaStream_t s) {
  k_scale_vals<<<grid_cap(nnz / 8), 256, 0, s>>>(nrows, rp, col, val, D_r, D_c, transposed, out64, out32);
}

__global__ void k_scale_vec(int len, const double* d, const double* v, double* out64, float* out32) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < len; i += gridDim.x * blockDim.x) {
    const double o = d[i] * v[i];
    out64[i] = o;
    if (out32) out32[i] = (float)o;
  }
}
void launch_scale_vec(int len, const double* d, const double* v, double* out64, float* out32,
                      cudaStream_t s) {
  k_scale_vec<<<grid_cap(len), 256, 0, s>>>(len, d, v, out64, out32);
}

// partials[block][8]: sums of b^2, c^2, b~^2, c~^2, min(0, c~)^2, three zeros
__global__ void __launch_bounds__(256) k_norms(int m, int n, const double* __restrict__ b,
                                               const double* __restrict__ c,
                                               const double* __restrict__ b_t,
                                               const double* __restrict__ c_t, double* partials) {
  __shared__ double red[8 * 8];
  double v[8] = {};
  const int step = gridDim.x * blockDim.x, t = blockIdx.x * blockDim.x + threadIdx.x;
  for (int i = t; i < m; i += step) {
    const double p = b[i], q = b_t[i];
    v[0] += p * p;
    v[2] += q * q;
  }
  for (int j = t; j < n; j += step) {
    const double p = c[j], q = c_t[j], r = min0(q);
    v[1] += p * p;
    v[3] += q * q;
    v[4] += r * r;
  }
  block_sum_scatter<256, 8>(v, red, partials + 8 * (size_t)blockIdx.x);
}

// ---------------------------------------------------------------------------
// power iteration on A~^T A~ (float64): u = A~ w, then w <- (A~^T u) / |w| in
// place with v . w and |w|^2, v = w / |w| of the step before.  The factor is
// applied a kernel late, so the last block of the next k_pow_Av adds a step's
// block sums (loads, a tree, a root, two divisions: 4 us, the power-law LP's
// steps 83 -> 79 us) while the others multiply.  Both kernels are launched with
// programmatic dependent launch and wait on entry, so each launch is set up
// while the previous kernel drains.
// ---------------------------------------------------------------------------
__global__ void k_pow_init(int n, double* w, PowerState* ps, int max_iter, double rel_tol) {
  const double v0 = 1.0 / sqrt((double)n);
  for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < n; j += gridDim.x * blockDim.x) w[j] = v0;
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    ps->lam = 0.0;
    ps->lam_prev = 0.0;
    ps->inv_norm = 1.0;
    ps->k = 0;
    ps->max_iter = max_iter;
    ps->stopped = (max_iter <= 0 || n == 0) ? 1 : 0;
    ps->ticket = 0;
    ps->rel_tol = rel_tol;
  }
}
void launch_pow_init(int n, double* w, PowerState* ps, int max_iter, double rel_tol,
                     cudaStream_t s) {
  k_pow_init<<<grid_cap(n), 256, 0, s>>>(n, w, ps, max_iter, rel_tol);
}

struct PowAvEpi {
  double* u;
  __device__ __forceinline__ void row(int r, const double (&s)[1], int) { u[r] = s[0]; }
};

// ends the step whose nparts block sums are in `partials`; one block
template <int BLOCK>
__device__ __forceinline__ void pow_step(PowerState* ps, const double* partials, int nparts) {
  __shared__ double red[2 * (BLOCK / 32)], tot[2];
  parts_sum<BLOCK, 2>(partials, nparts, nullptr, 0, tot, red);
  if (threadIdx.x != 0) return;
  const double lam = tot[0], nw = sqrt(tot[1]);
  ps->k += 1;
  ps->lam = lam;
  ps->inv_norm = nw == 0.0 ? 0.0 : 1.0 / nw;
  bool stop = nw == 0.0 || ps->k >= ps->max_iter;
  if (nw != 0.0) {
    stop = stop || (ps->k > 1 && fabs(lam - ps->lam_prev) <= ps->rel_tol * lam);
    ps->lam_prev = lam;
  }
  if (stop) ps->stopped = 1;
}
// the last step of power_max_iter
__global__ void __launch_bounds__(256) k_pow_end(PowerState* ps, const double* partials, int nparts) {
  if (!ps->stopped) pow_step<256>(ps, partials, nparts);
}

template <int BLOCK, int E>
__global__ void __launch_bounds__(BLOCK) k_pow_Av(SchedView S, const int32_t* rp, const int32_t* col,
                                                 const double* val, const double* w, double* u,
                                                 PowerState* ps, const double* partials, int nparts) {
  pdl_enter();
  if (ps->stopped) return;
  if (nparts && blockIdx.x == gridDim.x - 1) pow_step<BLOCK>(ps, partials, nparts);
  extern __shared__ __align__(16) unsigned char smem[];
  PowAvEpi epi{u};
  Gather<double, 1> g{{w}};
  run_sched<double, 1, BLOCK, E>(S, rp, col, val, g, epi, smem);
}

struct PowEpi {
  double* w;
  double inv, lam, nw2;
  double* split_q;
  __device__ __forceinline__ double load(int j) const { return w[j]; }
  __device__ __forceinline__ void apply(int j, double old, double s) {
    const double wn = s * inv;
    w[j] = wn;
    lam += (old * inv) * wn;
    nw2 += wn * wn;
  }
  __device__ __forceinline__ void row(int j, const double (&s)[1], int group) {
    if (group < 0) {
      apply(j, load(j), s[0]);
    } else {
      const double v = w[j] * inv, wn = s[0] * inv;
      w[j] = wn;
      split_q[2 * group] = v * wn;
      split_q[2 * group + 1] = wn * wn;
    }
  }
};

template <int BLOCK, int E>
__global__ void __launch_bounds__(BLOCK) k_pow_ATu(SchedView S, const int32_t* rp, const int32_t* col,
                                                  const double* val, const double* u, double* w,
                                                  double* partials, const PowerState* ps) {
  pdl_enter();
  if (ps->stopped) return;
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ double red[2 * (BLOCK / 32)];
  PowEpi epi{w, ps->inv_norm, 0.0, 0.0, partials + 2 * (size_t)gridDim.x};
  Gather<double, 1> g{{u}};
  run_sched<double, 1, BLOCK, E>(S, rp, col, val, g, epi, smem);
  double vv[2] = {epi.lam, epi.nw2};
  block_sum_scatter<BLOCK, 2>(vv, red, partials + 2 * (size_t)blockIdx.x);
}

void launch_pow_Av(const SchedView& S, const int32_t* rp, const int32_t* col, const double* val,
                   const double* w, double* u, PowerState* ps, const double* partials, int nparts,
                   const Launch& L, cudaStream_t s) {
  PDHG_DISPATCH_FIXED(S.e, launch_pdl(k_pow_Av<kBlock, E_>, L.grid, kBlock, L.smem, s, S, rp, col, val, w,
                                      u, ps, partials, nparts));
}
void launch_pow_ATu(const SchedView& S, const int32_t* rp, const int32_t* col, const double* val,
                    const double* u, double* w, double* partials, const PowerState* ps, const Launch& L,
                    cudaStream_t s) {
  PDHG_DISPATCH_FIXED(S.e, launch_pdl(k_pow_ATu<kBlock, E_>, L.grid, kBlock, L.smem, s, S, rp, col, val, u,
                                      w, partials, ps));
}
void launch_pow_end(PowerState* ps, const double* partials, int nparts, cudaStream_t s) {
  k_pow_end<<<1, 256, 0, s>>>(ps, partials, nparts);
}
template <int E>
static const void* pow_kernel(bool at) {
  return at ? (const void*)k_pow_ATu<kBlock, E> : (const void*)k_pow_Av<kBlock, E>;
}
int pow_occupancy(bool at, int e, size_t smem) {
  const void* f = e == kSliced ? pow_kernel<kSliced>(at) : pow_kernel<kFixedE>(at);
  int nb = 0;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, f, kBlock, smem);
  return nb < 1 ? 1 : nb;
}

// the norms from k_norms' partials (a fixed order), then the scalars of the
// solve; one block of 256
__global__ void k_init_scalars(Scalars* sc, const double* partials, int grid, const PowerState* ps,
                               double eta_safety) {
  __shared__ double sums[8], red[8 * 8];
  parts_sum<256, 8>(partials, grid, nullptr, 0, sums, red);
  if (threadIdx.x != 0) return;
  const double smax = sqrt(fmax(ps->lam, 0.0));
  sc->eta = smax > 0.0 ? eta_safety / smax : 1.0;
  const double nb = sqrt(sums[2]), nc = sqrt(sums[3]);
  sc->omega = (nb > 0.0 && nc > 0.0) ? nc / nb : 1.0;
  sc->tau = sc->eta / sc->omega;
  sc->sigma = sc->eta * sc->omega;
  sc->norm_b = sqrt(sums[0]);
  sc->norm_c = sqrt(sums[1]);
  const double w2 = sc->omega * sc->omega;
  sc->kkt_last = sqrt(w2 * sums[2] + sums[4] / w2);
  sc->kkt_prev = sc->kkt_last;
}
__global__ void k_recip(const double* __restrict__ in, double* out, int64_t len) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < len;
       i += (int64_t)gridDim.x * blockDim.x)
    out[i] = 1.0 / in[i];
}
void launch_recip(const double* in, double* out, int64_t len, cudaStream_t s) {
  const int64_t g = std::min<int64_t>(std::max<int64_t>((len + 255) / 256, 1), 4096);
  k_recip<<<(int)g, 256, 0, s>>>(in, out, len);
}

void launch_init_scalars(Scalars* sc, int m, int n, const double* b, const double* c,
                         const double* b_t, const double* c_t, double* partials,
                         const PowerState* ps, double eta_safety, cudaStream_t s) {
  const int grid = grid_cap(std::max(m, n), 1024, 256);
  k_norms<<<grid, 256, 0, s>>>(m, n, b, c, b_t, c_t, partials);
  k_init_scalars<<<1, 256, 0, s>>>(sc, partials, grid, ps, eta_safety);
}

// shared memory limit for the power-iteration tile kernels
cudaError_t configure_setup_kernels(size_t max_smem) {
  cudaError_t e = cudaSuccess;
  for (const void* f : {pow_kernel<kFixedE>(false), pow_kernel<kFixedE>(true), pow_kernel<kSliced>(false),
        pow_kernel<kSliced>(true)}) {
    cudaFuncAttributes a;
    cudaError_t r = cudaFuncGetAttributes(&a, f);
    if (r == cudaSuccess)
      r = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               (int)(max_smem - a.sharedSizeBytes));
    if (r != cudaSuccess) e = r;
  }
  return e;
}

// ---------------------------------------------------------------------------
// window words of a segmented schedule: one thread per (whole-row tile,
// thread window); the row of the window's first nonzero by binary search over
// the tile's rows, then the row ends inside the window
// ---------------------------------------------------------------------------
template <int E>
__global__ void k_window_words(const Tile* __restrict__ tiles, int ntiles,
                               const int32_t* __restrict__ rp,
                               typename WindowWord<E>::type* __restrict__ wd) {
  constexpr int e = E;
  const int64_t total = (int64_t)ntiles * kBlock;
  for (int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; idx < total;
       idx += (int64_t)gridDim.x * blockDim.x) {
    const int t = (int)(idx / kBlock), th = (int)(idx % kBlock);
    const Tile tl = tiles[t];
    if (tl.split >= 0 || tl.nz_begin == tl.nz_end) continue;
    const int w0 = (tl.nz_begin & ~3) + th * e;
    const int k0 = max(w0, tl.nz_begin), k1 = min(w0 + e, tl.nz_end);
    typename WindowWord<E>::type word = 0;
    if (k0 < k1) {
      int lo = tl.row_begin, hi = tl.row_end;  // rp[lo] <= k0 < rp[hi]
      while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (rp[mid] <= k0) lo = mid; else hi = mid;
      }
      uint64_t mask = 0;
      int r = lo, next_end = rp[lo + 1];
      for (int k = k0; k < k1; ++k)
        if (k + 1 == next_end) {
          mask |= 1ull << (k - w0);
          if (++r < tl.row_end) next_end = rp[r + 1];
        }
      word = window_word<E>(lo - tl.row_begin, rp[lo] < k0, mask);
    }
    wd[tl.word0 + th] = word;
  }
}

void launch_window_words(const Tile* tiles, int ntiles, const int32_t* rp, int e, uint32_t* wd,
                         cudaStream_t s) {
  if (ntiles <= 0) return;
  const int g = grid_cap((int64_t)ntiles * kBlock);
  if (e == 32)
    k_window_words<32><<<g, 256, 0, s>>>(tiles, ntiles, rp, reinterpret_cast<uint64_t*>(wd));
  else if (e == 16)
    k_window_words<16><<<g, 256, 0, s>>>(tiles, ntiles, rp, wd);
  else
    k_window_words<8><<<g, 256, 0, s>>>(tiles, ntiles, rp, wd);
}

}  // namespace pdhg
