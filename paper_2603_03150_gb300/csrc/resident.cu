// Solves of LPs that fit on chip: a thread-block cluster per LP runs whole
// solves (half-steps, evaluation, float64 check, restart) with the iterate in
// shared memory and no kernel launch between iterations; the power iteration
// of the set-up and the conjugate gradients of the adjoint run the same way.
// The layout and the device helpers are in resident.cuh.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <functional>
#include <new>
#include <numeric>
#include <vector>

#include "context.h"
#include "dispatch.cuh"
#include "eval_rule.cuh"
#include "resident.cuh"
#include "resident_host.h"

namespace pdhg {

// ---------------------------------------------------------------------------
// layout build (device; one block per LP and matrix sorts and cuts the slices,
// then a warp per slice fills it)
// ---------------------------------------------------------------------------
static __global__ void __launch_bounds__(256) k_res_sort(ResBuild B) {
  constexpr int kBins = kResMid + 2;  // lengths 0..kResMid, and the longer rows
  __shared__ int cursor[kBins];
  __shared__ int n_long, n_mid, longest;
  __shared__ long long carry;
  __shared__ int wsum[8];
  const int l = blockIdx.x >> 1, side = blockIdx.x & 1;
  ResLp& lp = B.lp[l];
  const int N = side ? lp.n : lp.m, C = lp.C, lg1 = side ? lp.lg_t : lp.lg_a, per = 32 >> lg1;
  const int64_t off = side ? lp.n_off : lp.m_off;
  const int32_t* rp = (side ? B.t_rp : B.a_rp) + off;
  uint16_t* ord = (side ? B.ord_n : B.ord_m) + off;
  uint16_t* pos = (side ? B.pos_n : B.pos_m) + off;
  ResSlice* sl = (side ? B.t_sl : B.a_sl) + off;
  const int tid = threadIdx.x, lane = tid & 31;
  for (int b = tid; b < kBins; b += 256) cursor[b] = 0;
  if (tid == 0) longest = 0;
  __syncthreads();
  int most = 0;
  for (int i = tid; i < N; i += 256) {
    const int len = rp[i + 1] - rp[i];
    most = max(most, len);
    atomicAdd(cursor + min(len, kBins - 1), 1);
  }
  atomicMax(&longest, most);
  __syncthreads();
  if (tid == 0) atomicMax(B.longest, longest);
  if (tid == 0) {  // longest first
    int run = 0, mid = 0;
    for (int b = kBins - 1; b >= 0; --b) {
      const int h = cursor[b];
      cursor[b] = run;
      run += h;
      if (b == kBins - 1) n_long = h;
      else if (b > kResShort) mid += h;
    }
    n_mid = mid;
    carry = 0;
  }
  __syncthreads();
  if (tid < 32) {  // stable ranks, 32 rows at a time
    int bin = lane < N ? min(rp[lane + 1] - rp[lane], kBins - 1) : -1;
    for (int base = 0; base < N; base += 32) {
      const int i = base + lane, nx = i + 32;
      const int next = nx < N ? min(rp[nx + 1] - rp[nx], kBins - 1) : -1;
      const unsigned peers = __match_any_sync(0xffffffffu, bin);
      const int first = bin >= 0 ? cursor[bin] : 0;
      __syncwarp();
      if (bin >= 0) {
        if (lane == __ffs(peers) - 1) cursor[bin] = first + __popc(peers);
        const int p = first + __popc(peers & ((1u << lane) - 1u));
        ord[p] = (uint16_t)i;
        pos[i] = (uint16_t)p;
      }
      __syncwarp();
      bin = next;
    }
  }
  __syncthreads();
  const int sL = n_long, sM = (n_mid + 3) / 4, n1 = N - n_long - n_mid, sS = (n1 + per - 1) / per;
  const int S = sL + sM + sS;
  for (int base = 0; base < S; base += 256) {
    const int s = base + tid;
    ResSlice d{0, 0, 0, 0};
    int w = 0;
    if (s < S) {
      const int r = s % C;
      auto mine = [&](int x) { return (x + C - 1 - r) / C; };  // slices of CTA r in [0, x)
      int lg, rows;
      if (s < sL) {
        lg = 5, rows = 1, d.p0 = s;
      } else if (s < sL + sM) {
        lg = 3, d.p0 = n_long + 4 * (s - sL), rows = min(4, n_long + n_mid - d.p0);
      } else {
        lg = lg1, d.p0 = n_long + n_mid + per * (s - sL - sM), rows = min(per, N - d.p0);
      }
      const int c1 = mine(min(s, sL)), c2 = mine(min(s, sL + sM)) - mine(min(s, sL)),
                c3 = mine(s) - mine(min(s, sL + sM));
      d.loc = c1 + 4 * c2 + per * c3;
      const int i = ord[d.p0], len = rp[i + 1] - rp[i];  // the slice's longest row
      w = (len + (1 << lg) - 1) >> lg;
      d.wgr = w | (lg << 16) | (rows << 20);
    }
    int incl = w;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int t = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += t;
    }
    if (lane == 31) wsum[tid >> 5] = incl;
    __syncthreads();
    int before = 0;
    for (int q = 0; q < (tid >> 5); ++q) before += wsum[q];
    if (s < S) {
      d.off = (int32_t)((carry + before + incl - w) * 32);
      sl[s] = d;
    }
    __syncthreads();
    if (tid == 255) carry += before + incl;
    __syncthreads();
  }
  if (tid == 0) {
    (side ? lp.t_slices : lp.a_slices) = S;
    B.elems[2 * l + side] = carry * 32;
  }
}

static __global__ void __launch_bounds__(256) k_res_fill(ResFill F, int count) {
  const int lane = threadIdx.x & 31;
  for (int q = blockIdx.y; q < 2 * count; q += gridDim.y) {  // (a grid has at most 65535 in y)
    const int l = q >> 1, side = q & 1;
    const ResLp lp = F.lp[l];
    const int64_t off = side ? lp.n_off : lp.m_off, coff = side ? lp.m_off : lp.n_off;
    const int32_t* rp = (side ? F.t_rp : F.a_rp) + off;
    const int32_t* col = side ? F.t_col : F.a_col;
    const double* val = side ? F.t_val : F.a_val;
    const int32_t* src = side ? F.t_src : F.a_src;
    const uint16_t* ord = (side ? F.ord_n : F.ord_m) + off;
    const uint16_t* pos = (side ? F.pos_m : F.pos_n) + coff;
    const ResSlice* sl = (side ? F.t_sl : F.a_sl) + off;
    const int64_t el = side ? lp.t_el : lp.a_el;
    uint16_t* oc = side ? F.t_c : F.a_c;
    double* ov = side ? F.t_v : F.a_v;
    float* of = side ? F.t_f : F.a_f;
    const uint16_t dummy = (uint16_t)(side ? lp.m : lp.n);
    const int S = side ? lp.t_slices : lp.a_slices;
    for (int s = blockIdx.x * 8 + (threadIdx.x >> 5); s < S; s += gridDim.x * 8) {
      const ResSlice d = sl[s];
      const int lg = res_lg(d.wgr), G = 1 << lg, row = lane >> lg, gl = lane & (G - 1);
      int b = 0, len = 0;
      if (row < res_rows(d.wgr)) {
        const int i = ord[d.p0 + row];
        b = rp[i];
        len = rp[i + 1] - b;
      }
      for (int k = 0; k < res_steps(d.wgr); ++k) {
        const int j = k * G + gl;
        uint16_t c = dummy;
        double v = 0.0;
        if (j < len) {
          v = val[src ? src[b + j] : b + j];
          if (oc) c = pos[col[b + j] - coff];
        }
        const int64_t at = el + d.off + k * 32 + lane;
        if (oc) oc[at] = c;
        ov[at] = v;
        if (of) of[at] = (float)v;
      }
    }
  }
}

void launch_res_sort(const ResBuild& B, int count, cudaStream_t s) {
  k_res_sort<<<2 * count, 256, 0, s>>>(B);
}
void launch_res_fill(const ResFill& F, int count, int max_slices, cudaStream_t s) {
  k_res_fill<<<dim3(std::min((max_slices + 7) / 8, 64), std::min(2 * count, 65535)), 256, 0, s>>>(F, count);
}

// ---------------------------------------------------------------------------
// power iteration on A~^T A~ (float64): u = A~w to every CTA's Y, then
// w <- (A~^T u) / |w| to every CTA's X with v . w and |w|^2, v = w / |w|.
// The vectors travel without the factor, so a step's sums (block, cluster, a
// root and a division: 1.3 us) are added by two warps while the others multiply
// by A~, and are needed only behind it.  They end an iteration that has begun:
// its first half-step is dropped.  An iteration of the LP 200 x 500, clusters of
// 4: 4.3 -> 2.7 us.
// ---------------------------------------------------------------------------
struct ResPower {
  const ResLp* lp;
  const int32_t* list;
  const ResSlice *a_sl, *t_sl;
  const uint16_t *a_col, *t_col;
  const double *a_val, *t_val;
  PowerState* ps;
  int max_iter;
  double rel_tol;
  unsigned long long wait_ns;
  uint32_t tx_extra;
  int32_t* err;  // 1 once a wait between CTAs ran out
};
template <int C>
__global__ void __launch_bounds__(kResThreads) k_res_power(ResPower A) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int l = A.list[blockIdx.x / C];
  const ResLp lp = A.lp[l];
  const ResSmem L = res_smem(lp.m, lp.n, lp.own_m, lp.own_n, 0, 0, 8);
  const ResCluster<C> cl(smem);
  double* X = reinterpret_cast<double*>(smem + L.X);
  double* Y = reinterpret_cast<double*>(smem + L.Y);
  const int tid = threadIdx.x;
  const ResMat Mt(A.t_sl + lp.n_off, A.t_col + lp.t_el, lp.t_slices, cl.rank, C);
  const ResMat Ma(A.a_sl + lp.m_off, A.a_col + lp.a_el, lp.a_slices, cl.rank, C);
  const double *tv = A.t_val + lp.t_el, *av = A.a_val + lp.a_el;
  const double v0 = 1.0 / sqrt((double)lp.n);
  for (int j = tid; j < lp.n; j += kResThreads) X[j] = v0;
  if (tid == 0) {
    X[lp.n] = 0.0;
    Y[lp.m] = 0.0;
  }
  ResExchange<C> ex(cl, L, smem, A.wait_ns, (uint32_t)lp.n * 8u, (uint32_t)lp.m * 8u, 2, 2,
                    A.tx_extra, res_idle(Ma, Mt));
  double lam = 0.0, lam_prev = 0.0, inv = A.max_iter > 0 ? 1.0 : 0.0;
  int k = 0;  // steps whose w has been computed
  cl.sync();
  for (bool stop = A.max_iter <= 0; !stop;) {
    const bool more = k < A.max_iter;
    if (more)
      Ma.template each<C>([&](const ResSlice& s, int row) {
        const double* const buf[1] = {X};
        double u[1] = {0.0};
        res_dot<1, false>(s, av, Ma.col, buf, u);
        if (row >= 0) ex.send_y(s.p0 + row, u[0]);
      });
    if (k > 0) {  // the sums of step k
      double t[2][2];
      stop = ex.template sum_end<2>((k - 1) & 1, ((k - 1) >> 1) & 1, t, [&](int which, double v, double (&o)[2]) {
        if (which == 0) {  // lam, and whether it has settled
          o[0] = v;
          o[1] = k > 1 && fabs(v - lam_prev) <= A.rel_tol * v ? 1.0 : 0.0;
        } else {  // |w|^2 = 0, 1 / |w|
          o[0] = v == 0.0 ? 1.0 : 0.0;
          o[1] = v == 0.0 ? 0.0 : 1.0 / sqrt(v);
        }
      });
      const bool zero = __double_as_longlong(t[1][0]) != 0;
      lam = t[0][0];
      inv = t[1][1];
      if (!zero) lam_prev = lam;
      stop = stop || zero || __double_as_longlong(t[0][1]) != 0 || !more;
    }
    if (more) ex.wait(1);  // (what is under way to this CTA arrives before it leaves)
    if (stop) break;
    double q[2] = {0.0, 0.0};
    Mt.template each<C>([&](const ResSlice& s, int row) {
      const double* const buf[1] = {Y};
      double w[1] = {0.0};
      res_dot<1, false>(s, tv, Mt.col, buf, w);
      if (row < 0) return;
      const double v = X[s.p0 + row] * inv, wn = w[0] * inv;
      q[0] += v * wn;
      q[1] += wn * wn;
      ex.send_x(s.p0 + row, wn);
    });
    ex.template sum_begin<2>(q, k & 1);
    k += 1;
    ex.wait(0);
    ex.next();
  }
  if (ex.finish()) {
    if (tid == 0) atomicExch(A.err, 1);
    return;
  }
  if (cl.rank == 0 && tid == 0) {
    PowerState p{};
    p.lam = lam;
    p.lam_prev = lam_prev;
    p.inv_norm = inv;
    p.k = k;
    p.max_iter = A.max_iter;
    p.stopped = 1;
    p.rel_tol = A.rel_tol;
    A.ps[l] = p;
  }
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
struct ResData {
  ResLp* lp = nullptr;
  int32_t* list = nullptr;
  ResSlice *a_sl = nullptr, *t_sl = nullptr;
  uint16_t *ord_m = nullptr, *ord_n = nullptr, *pos_m = nullptr, *pos_n = nullptr;
  uint16_t *a_col = nullptr, *t_col = nullptr;
  double *a_val = nullptr, *t_val = nullptr;
  float *a_f = nullptr, *t_f = nullptr;
  int32_t* active = nullptr;  // [0] LPs not finished, [1] a wait ran out
  int max_slices = 1;
  std::vector<ResGroup> groups;
  ResStreams side;
};
static ResData* res_of(const pdhg_ctx* ctx) { return static_cast<ResData*>(ctx->resident); }

static const void* solve_kernel(const pdhg_ctx* ctx, int C) {
  const bool hal = ctx->opt.method == 1;
  return ctx->mixed ? res_solve_kernel<float>(C, hal) : res_solve_kernel<double>(C, hal);
}
static const void* power_kernel(int C) {
  const void* f = nullptr;
  RES_DISPATCH_C(C, f = (const void*)k_res_power<C_>);
  return f;
}

// the kernel may run with `smem` bytes in clusters of C (its limits are raised)
bool res_fits(const void* f, int C, size_t smem, size_t smem_optin) {
  if (set_max_dyn_smem(f, smem_optin) != cudaSuccess) return false;
  cudaFuncAttributes a;
  if (cudaFuncGetAttributes(&a, f) != cudaSuccess || smem + a.sharedSizeBytes > smem_optin) return false;
  if (C == 1) return true;
  if (C > 8 && cudaFuncSetAttribute(f, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess)
    return false;
  cudaLaunchAttribute attr;
  const cudaLaunchConfig_t cfg = res_config(C, 1, smem, nullptr, &attr);
  int n = 0;
  const bool ok = cudaOccupancyMaxActiveClusters(&n, f, &cfg) == cudaSuccess && n >= 1;
  cudaGetLastError();
  return ok;
}

void resident_free(pdhg_ctx* ctx) {
  ResData* d = res_of(ctx);
  if (!d) return;
  d->side.free();
  delete d;
  ctx->resident = nullptr;
}

static ResSmem solve_smem(const pdhg_ctx* ctx, int m, int n, int C) {
  const bool hal = ctx->opt.method == 1;
  return res_smem(m, n, res_own(m, C), res_own(n, C), hal ? 6 : 4, hal ? 4 : 2, ctx->mixed ? 4 : 8);
}

// The cluster size of every LP: for each of several shares of the batch's work
// that a CTA takes at most, the schedule (largest first, each cluster on the
// SMs that are free first) is played through and the shortest kept.  A CTA gets
// at least min_ops operations of an iteration and an LP room for its vectors;
// empty where an LP fits in no cluster.  512 float64 LPs: shares of 1/8 / 1/4 /
// 1/2 / 1 of an SM's mean 76 / 53 / 47 / 46 ms; 64 LPs of 2000 x 5000 on 152
// SMs: clusters of 4 run in two waves (11.1 ms), of 2 in one.
std::vector<int> res_clusters(const pdhg_ctx* ctx, const std::vector<double>& ops, double min_ops,
                              const std::function<bool(int, int)>& fits) {
  const int count = (int)ops.size();
  std::vector<int> least((size_t)count), order((size_t)count), best;
  double total = 0.0;
  for (int l = 0; l < count; ++l) {
    int c = 1;
    while (c < kResMaxC && !fits(l, c)) c *= 2;
    if (!fits(l, c)) return {};
    least[l] = c;
    total += ops[l];
  }
  std::iota(order.begin(), order.end(), 0);
  double shortest = 0.0;
  for (double f = 0.25; f < 5.0; f *= 1.41421356) {
    const double share = std::max(f * total / ctx->nsm, min_ops);
    std::vector<int> C(least);
    for (int l = 0; l < count; ++l)
      while (C[l] < kResMaxC && ops[l] > share * C[l]) C[l] *= 2;
    std::sort(order.begin(), order.end(), [&](int a, int b) {
      if (C[a] != C[b]) return C[a] > C[b];
      if (ops[a] != ops[b]) return ops[a] > ops[b];
      return a < b;
    });
    std::vector<double> busy((size_t)ctx->nsm, 0.0);  // ascending
    for (int l : order) {
      // clocks of an iteration: 2 operations per clock and SM, and the exchanges
      const int c = std::min(C[l], ctx->nsm);
      const double t = ops[l] / (2.0 * C[l]) + (C[l] > 1 ? 2000.0 : 1500.0);
      const double end = busy[c - 1] + t;
      busy.erase(busy.begin(), busy.begin() + c);
      busy.insert(std::upper_bound(busy.begin(), busy.end(), end), (size_t)c, end);
    }
    if (best.empty() || busy.back() < shortest) {
      shortest = busy.back();
      best = C;
    }
  }
  return best;
}

// the LPs by cluster size, then work (a launch group is a run of one size)
std::vector<int32_t> res_order(const std::vector<ResLp>& lps, const std::vector<double>& ops) {
  std::vector<int32_t> list(lps.size());
  std::iota(list.begin(), list.end(), 0);
  std::sort(list.begin(), list.end(), [&](int a, int b) {
    if (lps[a].C != lps[b].C) return lps[a].C > lps[b].C;
    if (ops[a] != ops[b]) return ops[a] > ops[b];
    return a < b;
  });
  return list;
}

// Chooses the cluster size of every LP and builds the layout; leaves
// ctx->resident NULL where the LPs do not fit on chip, options ask for the tile
// kernels' own paths or there is no memory for it.
static pdhg_status res_build(pdhg_ctx* ctx) {
  const pdhg_options& o = ctx->opt;
  // A float32-mixed solve of one LP keeps the tile kernels' order of addition:
  // its float64 solution is that of float32 iterates, which differ by 1e-6
  // between orders, and a program that stores or compares such solutions would
  // see it.
  if (ctx->mixed && !ctx->batch) return PDHG_OK;
  if (o.tile_nnz != 0 || o.spmv_layout != 0 || o.panel_width != 0 || o.kernel_timing != 0 ||
      o.step_rule != 0 || (ctx->batch && o.persistent != 0))
    return PDHG_OK;
  const int count = ctx->count;
  std::vector<ResLp> lps((size_t)count);
  std::vector<double> ops((size_t)count);
  for (int l = 0; l < count; ++l) {
    ResLp& p = lps[l];
    p = ResLp{};
    p.m_off = ctx->batch ? ctx->h_m_off[l] : 0;
    p.n_off = ctx->batch ? ctx->h_n_off[l] : 0;
    p.m = ctx->batch ? (int)(ctx->h_m_off[l + 1] - p.m_off) : ctx->m;
    p.n = ctx->batch ? (int)(ctx->h_n_off[l + 1] - p.n_off) : ctx->n;
    const int64_t z = (int64_t)ctx->h_a_rp[p.m_off + p.m] - ctx->h_a_rp[p.m_off];
    if (p.m > 65534 || p.n > 65534 || z > kResMaxNnz) return PDHG_OK;
    ops[l] = 2.0 * (double)z + 3.0 * p.n + 7.0 * p.m;
  }
  auto fits = [&](int l, int c) {
    const size_t need = std::max<size_t>(
        solve_smem(ctx, lps[l].m, lps[l].n, c).total,
        res_smem(lps[l].m, lps[l].n, res_own(lps[l].m, c), res_own(lps[l].n, c), 0, 0, 8).total);
    return need + 2048 <= ctx->smem_optin;  // the kernels' static shared memory
  };
  const std::vector<int> Cs = res_clusters(ctx, ops, ctx->mixed ? kResMinOps32 : kResMinOps64, fits);
  if (Cs.empty()) return PDHG_OK;
  for (int l = 0; l < count; ++l) {
    ResLp& q = lps[l];
    const int64_t z = (int64_t)ctx->h_a_rp[q.m_off + q.m] - ctx->h_a_rp[q.m_off];
    q.C = Cs[l];
    q.lg_a = res_lanes(q.m, z, q.C);
    q.lg_t = res_lanes(q.n, z, q.C);
  }
  bool use[5] = {};
  // the cluster sizes the device runs (16 may not be available)
  for (int l = 0; l < count; ++l) use[(int)std::lround(std::log2(lps[l].C))] = true;
  for (int q = 0; q < 5; ++q) {
    if (!use[q]) continue;
    const int C = 1 << q;
    size_t need = 0, needp = 0;
    for (const ResLp& p : lps)
      if (p.C == C) {
        need = std::max<size_t>(need, solve_smem(ctx, p.m, p.n, C).total);
        needp = std::max<size_t>(needp, res_smem(p.m, p.n, res_own(p.m, C), res_own(p.n, C), 0, 0, 8).total);
      }
    if (!res_fits(solve_kernel(ctx, C), C, need, ctx->smem_optin) ||
        !res_fits(power_kernel(C), C, needp, ctx->smem_optin))
      return PDHG_OK;
  }
  ResData* d = new (std::nothrow) ResData();
  if (!d) {
    set_error("out of host memory");
    return PDHG_OOM;
  }
  ctx->resident = d;
  const size_t m = (size_t)ctx->m, n = (size_t)ctx->n;
  CKS(dalloc(ctx, &d->lp, (size_t)count));
  CKS(dalloc(ctx, &d->list, (size_t)count));
  CKS(dalloc(ctx, &d->active, 2));
  CKS(dalloc(ctx, &d->a_sl, m));
  CKS(dalloc(ctx, &d->t_sl, n));
  CKS(dalloc(ctx, &d->ord_m, m));
  CKS(dalloc(ctx, &d->ord_n, n));
  CKS(dalloc(ctx, &d->pos_m, m));
  CKS(dalloc(ctx, &d->pos_n, n));
  long long* elems = nullptr;
  CKS(dalloc(ctx, &elems, 2 * (size_t)count));
  CK(cudaMemsetAsync(d->active, 0, 2 * sizeof(int32_t), ctx->stream));
  // launch groups by cluster size, the largest LPs first
  std::vector<int32_t> list = res_order(lps, ops);
  for (int i = 0; i < count; ++i) {
    ResLp& p = lps[list[i]];
    p.own_m = res_own(p.m, p.C);
    p.own_n = res_own(p.n, p.C);
    if (d->groups.empty() || d->groups.back().C != p.C) d->groups.push_back(ResGroup{p.C, i, 0});
    ResGroup& g = d->groups.back();
    g.count += 1;
    g.smem_solve = std::max<size_t>(g.smem_solve, solve_smem(ctx, p.m, p.n, p.C).total);
    g.smem_power =
        std::max<size_t>(g.smem_power, res_smem(p.m, p.n, p.own_m, p.own_n, 0, 0, 8).total);
  }
  CK(cudaMemcpyAsync(d->lp, lps.data(), sizeof(ResLp) * count, cudaMemcpyHostToDevice, ctx->stream));
  CK(cudaMemcpyAsync(d->list, list.data(), sizeof(int32_t) * count, cudaMemcpyHostToDevice, ctx->stream));
  ResBuild b{d->lp, ctx->a_rp, ctx->t_rp, d->a_sl, d->t_sl, d->ord_m, d->ord_n, d->pos_m, d->pos_n, elems,
             d->active};
  launch_res_sort(b, count, ctx->stream);
  std::vector<long long> el(2 * (size_t)count);
  CK(cudaMemcpyAsync(el.data(), elems, sizeof(long long) * el.size(), cudaMemcpyDeviceToHost, ctx->stream));
  CK(cudaMemcpyAsync(lps.data(), d->lp, sizeof(ResLp) * count, cudaMemcpyDeviceToHost, ctx->stream));
  int32_t longest = 0;
  CK(cudaMemcpyAsync(&longest, d->active, sizeof(longest), cudaMemcpyDeviceToHost, ctx->stream));
  CK(cudaStreamSynchronize(ctx->stream));
  if (longest > kResMaxRow) {
    resident_free(ctx);
    return PDHG_OK;
  }
  // A CTA without a slice of either matrix would have no warp that is held to the
  // others' phases.  (A CTA's share of the work is at least kResMinOps
  // operations, so every CTA of a cluster has slices.)
  for (const ResLp& p : lps)
    if (std::max(p.a_slices, p.t_slices) < p.C) {
      resident_free(ctx);
      return PDHG_OK;
    }
  int64_t ea = 0, et = 0;
  for (int l = 0; l < count; ++l) {
    lps[l].a_el = ea;
    lps[l].t_el = et;
    ea += el[2 * l];
    et += el[2 * l + 1];
    d->max_slices = std::max({d->max_slices, lps[l].a_slices, lps[l].t_slices});
  }
  CKS(dalloc(ctx, &d->a_col, (size_t)ea));
  CKS(dalloc(ctx, &d->t_col, (size_t)et));
  CKS(dalloc(ctx, &d->a_val, (size_t)ea));
  CKS(dalloc(ctx, &d->t_val, (size_t)et));
  if (ctx->mixed) {
    CKS(dalloc(ctx, &d->a_f, (size_t)ea));
    CKS(dalloc(ctx, &d->t_f, (size_t)et));
  }
  CK(cudaMemcpyAsync(d->lp, lps.data(), sizeof(ResLp) * count, cudaMemcpyHostToDevice, ctx->stream));
  launch_res_fill(ResFill{d->lp, ctx->a_rp, ctx->t_rp, ctx->a_col, ctx->t_col, ctx->a_val64,
                          ctx->t_val64, nullptr, nullptr, d->a_sl, d->t_sl, d->ord_m, d->ord_n,
                          d->pos_m, d->pos_n, d->a_col, d->t_col, d->a_val, d->t_val, d->a_f, d->t_f},
                  count, d->max_slices, ctx->stream);
  ctx->launches += 2;
  CK(cudaGetLastError());
  CK(d->side.make((int)d->groups.size()));
  CK(cudaStreamSynchronize(ctx->stream));  // the host vectors go out of scope
  return PDHG_OK;
}

pdhg_status resident_build(pdhg_ctx* ctx) {
  return if_room(ctx, [&] { return res_build(ctx); }, [&] { resident_free(ctx); });
}

pdhg_status resident_power(pdhg_ctx* ctx) {
  ResData* d = res_of(ctx);
  ResPower A{d->lp,    nullptr,  d->a_sl, d->t_sl, d->a_col, d->t_col,
             d->a_val, d->t_val, ctx->ps, ctx->opt.power_max_iter, ctx->opt.power_rel_tol,
             (unsigned long long)ctx->opt.wait_limit_ms * 1000000ull, res_tx_extra(ctx), d->active + 1};
  CKS(res_groups(ctx, d->groups, d->side, [&](const ResGroup& g, cudaStream_t s) {
    A.list = d->list + g.first;
    cudaLaunchAttribute attr;
    const cudaLaunchConfig_t cfg = res_config(g.C, g.count, g.smem_power, s, &attr);
    cudaError_t e = cudaSuccess;
    RES_DISPATCH_C(g.C, e = cudaLaunchKernelEx(&cfg, k_res_power<C_>, A));
    return e;
  }));
  int32_t err = 0;
  CK(cudaMemcpyAsync(&err, d->active + 1, sizeof(err), cudaMemcpyDeviceToHost, ctx->stream));
  CK(cudaStreamSynchronize(ctx->stream));
  if (err) {
    set_error("power iteration: a CTA waited longer than options.wait_limit_ms for another's vector");
    return PDHG_TIMEOUT;
  }
  return PDHG_OK;
}

template <typename T>
static pdhg_status res_solve(pdhg_ctx* ctx, const IterBuffers<T>& B, int32_t* active) {
  ResData* d = res_of(ctx);
  ResSolve<T> A{};
  A.lp = d->lp;
  A.a_sl = d->a_sl;
  A.t_sl = d->t_sl;
  A.a_col = d->a_col;
  A.t_col = d->t_col;
  A.ord_m = d->ord_m;
  A.ord_n = d->ord_n;
  if constexpr (sizeof(T) == 4) {
    A.a_val = d->a_f;
    A.t_val = d->t_f;
  } else {
    A.a_val = d->a_val;
    A.t_val = d->t_val;
  }
  A.a_val64 = d->a_val;
  A.t_val64 = d->t_val;
  A.B = B;
  A.active = active;
  A.slice_ns = 100000000ull;
  A.wait_ns = (unsigned long long)ctx->opt.wait_limit_ms * 1000000ull;
  A.tx_extra = res_tx_extra(ctx);
  A.err = d->active + 1;
  return res_groups(ctx, d->groups, d->side, [&](const ResGroup& g, cudaStream_t s) {
    A.list = d->list + g.first;
    return launch_res_solve<T>(A, g.C, g.count, g.smem_solve, ctx->opt.method == 1, s);
  });
}

// Runs every LP to its end.  Each launch ends by itself after its time slice;
// then the host reads how many LPs have not finished.
template <typename T>
pdhg_status resident_solve(pdhg_ctx* ctx, const IterBuffers<T>& B) {
  int32_t* active = res_of(ctx)->active;
  int32_t* left = reinterpret_cast<int32_t*>(ctx->h_sc[0]);  // pinned
  left[0] = ctx->count;
  left[1] = 0;
  CK(cudaMemcpyAsync(active, left, 2 * sizeof(int32_t), cudaMemcpyHostToDevice, ctx->stream));
  do {
    CKS(res_solve<T>(ctx, B, active));
    CK(cudaMemcpyAsync(left, active, 2 * sizeof(int32_t), cudaMemcpyDeviceToHost, ctx->stream));
    CK(cudaStreamSynchronize(ctx->stream));
    CK(cudaGetLastError());
    if (left[1]) {
      set_error("a CTA waited longer than options.wait_limit_ms for another's vector; the iterate "
                "is not meaningful");
      return PDHG_TIMEOUT;
    }
  } while (left[0] > 0);
  return PDHG_OK;
}
template pdhg_status resident_solve<float>(pdhg_ctx*, const IterBuffers<float>&);
template pdhg_status resident_solve<double>(pdhg_ctx*, const IterBuffers<double>&);

}  // namespace pdhg
