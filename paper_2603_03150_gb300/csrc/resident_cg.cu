// Conjugate gradients of the active-set polish and adjoint, on chip: a cluster
// per LP (resident.cuh) runs all steps of M_B^T M_B w = rhs with p and u = M_B p
// in shared memory.  B, the columns of positive x, is about a third of an LP's
// columns and p is zero off it, so the matrices are cut down to B first (the
// terms left out are exact zeros): a step takes 2 float64 operations per nonzero
// of B's columns and 5 per column of B.
#include <algorithm>
#include <cstring>
#include <new>

#include "resident_host.h"

namespace pdhg {

namespace {

// ---------------------------------------------------------------------------
// the matrices cut down to B: row pointers, columns (B's own numbering) and
// where each entry's values are
// ---------------------------------------------------------------------------
__global__ void k_sub_flags(int n, const double* __restrict__ mask, int32_t* flag) {
  for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < n; j += gridDim.x * blockDim.x)
    flag[j] = mask[j] != 0.0;
}

// columns of A in B: their list and lengths, and the entries of each row in B
__global__ void k_sub_count(int m, int n, const int32_t* __restrict__ a_rp,
                            const int32_t* __restrict__ a_col, const int32_t* __restrict__ t_rp,
                            const double* __restrict__ mask, const int32_t* __restrict__ idx,
                            int32_t* bcol, int32_t* t_len, int32_t* a_len) {
  const int step = gridDim.x * blockDim.x, t = blockIdx.x * blockDim.x + threadIdx.x;
  for (int j = t; j < n; j += step)
    if (mask[j] != 0.0) {
      bcol[idx[j]] = j;
      t_len[idx[j]] = t_rp[j + 1] - t_rp[j];
    }
  for (int i = t >> 3; i < m; i += step >> 3) {  // 8 lanes per row
    int c = 0;
    for (int k = a_rp[i] + (t & 7); k < a_rp[i + 1]; k += 8) c += mask[a_col[k]] != 0.0;
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) c += __shfl_down_sync(0xffu << (threadIdx.x & 24), c, o, 8);
    if ((t & 7) == 0) a_len[i] = c;
  }
}

__global__ void k_sub_fill(int m, int nb, const int32_t* __restrict__ a_rp,
                           const int32_t* __restrict__ a_col, const int32_t* __restrict__ t_rp,
                           const int32_t* __restrict__ t_col, const double* __restrict__ mask,
                           const int32_t* __restrict__ idx, const int32_t* __restrict__ bcol,
                           const int32_t* __restrict__ sa_rp, const int32_t* __restrict__ st_rp,
                           int32_t* sa_col, int32_t* sa_src, int32_t* st_col, int32_t* st_src) {
  const int step = gridDim.x * blockDim.x, t = blockIdx.x * blockDim.x + threadIdx.x;
  for (int q = t; q < nb; q += step) {
    const int j = bcol[q], s = t_rp[j], d = st_rp[q], len = t_rp[j + 1] - s;
    for (int e = 0; e < len; ++e) {
      st_col[d + e] = t_col[s + e];
      st_src[d + e] = s + e;
    }
  }
  for (int i = t; i < m; i += step) {
    int d = sa_rp[i];
    for (int k = a_rp[i]; k < a_rp[i + 1]; ++k) {
      const int j = a_col[k];
      if (mask[j] != 0.0) {
        sa_col[d] = idx[j];
        sa_src[d++] = k;
      }
    }
  }
}

// ---------------------------------------------------------------------------
struct ResCg {
  const ResLp* lp;      // n: the columns of B
  const int32_t* list;
  const ResSlice *a_sl, *t_sl;
  const uint16_t *a_col, *t_col, *ord_n;
  const double *a_val, *t_val;
  const int32_t* bcol;  // the column of each of B's columns
  const double* rhs;
  double* w;            // in: the start; out: the solution (B's columns only)
  int32_t* iters;
  double tol2;
  int max_iter;
  unsigned long long wait_ns;
  uint32_t tx_extra;
  int32_t* err;
};

// Bound by the float64 pipe with an SM per LP or more LPs than SMs, else by the
// latency of a pass over a slice, two exchanges of a vector and two sums per
// step.  64 LPs of 2000 x 5000: 8.8 us per step (676 steps of the adjoint in 5.9
// ms) against 57 us of four launches on the tile kernels; 5 LPs of 333 x 832:
// 6.0 us against 31.  With every warp taking the sums and quotients itself the
// same steps took 12.5 and 9 us.
template <int C>
__global__ void __launch_bounds__(kResThreads) k_res_cg(ResCg A) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int l = A.list[blockIdx.x / C];
  const ResLp lp = A.lp[l];
  const ResSmem L = res_smem(lp.m, lp.n, lp.own_m, lp.own_n, 0, 3, 8);
  const ResCluster<C> cl(smem);
  double* X = reinterpret_cast<double*>(smem + L.X);  // p
  double* Y = reinterpret_cast<double*>(smem + L.Y);  // u
  double* w = reinterpret_cast<double*>(smem + L.own_n);
  double* r = w + lp.own_n;
  double* qv = r + lp.own_n;
  const int tid = threadIdx.x;
  const ResMat Mt(A.t_sl + lp.n_off, A.t_col + lp.t_el, lp.t_slices, cl.rank, C);
  const ResMat Ma(A.a_sl + lp.m_off, A.a_col + lp.a_el, lp.a_slices, cl.rank, C);
  const double *tv = A.t_val + lp.t_el, *av = A.a_val + lp.a_el;
  const uint16_t* on = A.ord_n + lp.n_off;
  const int32_t* bcol = A.bcol + lp.n_off;
  ResExchange<C> ex(cl, L, smem, A.wait_ns, (uint32_t)lp.n * 8u, (uint32_t)lp.m * 8u, 2, 1,
                    A.tx_extra, res_idle(Ma, Mt));
  if (tid == 0) {
    X[lp.n] = 0.0;
    Y[lp.m] = 0.0;
  }
  cl.sync();  // every CTA has started
  // r = rhs - M_B^T M_B w0, p = r (an iteration of its own for the barriers)
  Mt.template each<C>([&](const ResSlice& s, int row) {
    if (row < 0) return;
    const double v = A.w[bcol[on[s.p0 + row]]];
    w[s.loc + row] = v;
    cl.push(L.X + (uint32_t)(s.p0 + row) * 8u, v);
  });
  cl.sync();
  auto product = [&]() {  // u = M_B p
    Ma.template each<C>([&](const ResSlice& s, int row) {
      const double* const buf[1] = {X};
      double u[1] = {0.0};
      res_dot<1, false>(s, av, Ma.col, buf, u);
      if (row >= 0) ex.send_y(s.p0 + row, u[0]);
    });
    ex.wait(1);
  };
  product();
  double q[2] = {0.0, 0.0};
  Mt.template each<C>([&](const ResSlice& s, int row) {
    const double* const buf[1] = {Y};
    double v[1] = {0.0};
    res_dot<1, false>(s, tv, Mt.col, buf, v);
    if (row < 0) return;
    const double b = A.rhs[bcol[on[s.p0 + row]]], rj = b - v[0];
    r[s.loc + row] = rj;
    q[0] += rj * rj;
    q[1] += b * b;
  });
  double t[2][3];
  ex.sum(q, 0, t, [&](int, double v, double (&o)[3]) {
    o[0] = v;
    o[1] = A.tol2 * v;
    o[2] = 0.0;
  });
  double rr = t[0][0];
  const double stop = t[1][1];
  int it = 0;
  bool done = rr <= stop || A.max_iter <= 0;
  if (!ex.ends(done)) {
    Mt.template each<C>([&](const ResSlice& s, int row) {
      if (row >= 0) ex.send_x(s.p0 + row, r[s.loc + row]);
    });
    ex.wait(0);
    double unused[1] = {0.0}, none[1][3];
    ex.sum(unused, 1, none, [](int, double, double (&o)[3]) { o[0] = o[1] = o[2] = 0.0; });
    ex.next();
    while (true) {
      product();
      q[0] = q[1] = 0.0;
      Mt.template each<C>([&](const ResSlice& s, int row) {
        const double* const buf[1] = {Y};
        double v[1] = {0.0};
        res_dot<1, false>(s, tv, Mt.col, buf, v);
        if (row < 0) return;
        qv[s.loc + row] = v[0];
        q[0] += X[s.p0 + row] * v[0];
      });
      ex.sum(q, 0, t, [&](int, double v, double (&o)[3]) {
        o[0] = v;
        o[1] = v > 0.0 ? rr / v : 0.0;
        o[2] = 0.0;
      });
      const double pq = t[0][0], alpha = t[0][1];
      double sq[1] = {0.0};
      Mt.template each<C>([&](const ResSlice& s, int row) {
        if (row < 0) return;
        const int k = s.loc + row;
        w[k] += alpha * X[s.p0 + row];
        const double rj = r[k] - alpha * qv[k];
        r[k] = rj;
        sq[0] += rj * rj;
      });
      it += 1;
      double b[1][3];
      ex.sum(sq, 1, b, [&](int, double v, double (&o)[3]) {
        o[0] = v;
        o[1] = rr > 0.0 ? v / rr : 0.0;
        o[2] = v <= stop || it >= A.max_iter || !(pq > 0.0) ? 1.0 : 0.0;
      });
      rr = b[0][0];
      const double beta = b[0][1];
      done = __double_as_longlong(b[0][2]) != 0;
      if (ex.ends(done)) break;
      Mt.template each<C>([&](const ResSlice& s, int row) {
        if (row >= 0) ex.send_x(s.p0 + row, r[s.loc + row] + beta * X[s.p0 + row]);
      });
      ex.wait(0);
      ex.next();
    }
  }
  if (ex.finish()) {
    if (tid == 0) atomicExch(A.err, 1);
  } else {
    Mt.template each<C>([&](const ResSlice& s, int row) {
      if (row >= 0) A.w[bcol[on[s.p0 + row]]] = w[s.loc + row];
    });
    if (cl.rank == 0 && tid == 0) A.iters[l] = it;
  }
}

const void* cg_kernel(int C) {
  const void* f = nullptr;
  RES_DISPATCH_C(C, f = (const void*)k_res_cg<C_>);
  return f;
}

size_t cg_smem(int m, int n, int C) {
  return res_smem(m, n, res_own(m, C), res_own(n, C), 0, 3, 8).total;
}

}  // namespace

struct ResCgData {
  ResLp* lp = nullptr;
  int32_t* list = nullptr;
  ResSlice *a_sl = nullptr, *t_sl = nullptr;
  uint16_t *ord_m = nullptr, *ord_n = nullptr, *pos_m = nullptr, *pos_n = nullptr;
  uint16_t *a_col = nullptr, *t_col = nullptr;
  double *val[2][2] = {};  // [scaled, original][A, A^T]
  int32_t *idx = nullptr, *bcol = nullptr, *len = nullptr, *scan = nullptr;
  int32_t *sa_rp = nullptr, *st_rp = nullptr, *sa_col = nullptr, *sa_src = nullptr, *st_col = nullptr,
          *st_src = nullptr;
  int32_t *iters = nullptr, *flags = nullptr;  // flags: [0] longest row, [1] a wait ran out
  long long* elems = nullptr;
  size_t cap = 0;
  bool ready = false, original = false;
  int max_slices = 1;
  std::vector<ResLp> lps;
  std::vector<ResGroup> groups;
  ResStreams side;
};

ResCgData* resident_cg_new() { return new (std::nothrow) ResCgData(); }
void resident_cg_free(ResCgData* d) {
  if (!d) return;
  d->side.free();
  delete d;
}
bool resident_cg_ready(const ResCgData* d) { return d && d->ready; }

// B = the columns with mask != 0, active[l] of them in LP l; not ready where the
// LPs are not solved on chip or there is no memory for the layout
static pdhg_status cg_layout(pdhg_ctx* ctx, ResCgData* d, const double* mask, const int32_t* active) {
  d->ready = d->original = false;
  if (!ctx->resident) return PDHG_OK;
  const int count = ctx->count, m = ctx->m, n = ctx->n;
  std::vector<double> ops((size_t)count);
  d->lps.assign((size_t)count, ResLp{});
  int64_t nb = 0;
  for (int l = 0; l < count; ++l) {
    ResLp& p = d->lps[l];
    p.m_off = ctx->h_m_off[l];
    p.m = (int)(ctx->h_m_off[l + 1] - p.m_off);
    p.n_off = nb;
    p.n = active[l];
    nb += active[l];
    // B's share of the nonzeros, and 5 operations per column
    const double z = (double)(ctx->h_a_rp[p.m_off + p.m] - ctx->h_a_rp[p.m_off]);
    const double nl = (double)(ctx->h_n_off[l + 1] - ctx->h_n_off[l]);
    ops[l] = 2.0 * z * p.n / nl + 5.0 * p.n;
  }
  const std::vector<int> Cs = res_clusters(ctx, ops, kResMinOps64, [&](int l, int c) {
    return cg_smem(d->lps[l].m, d->lps[l].n, c) + 2048 <= ctx->smem_optin;
  });
  if (Cs.empty()) return PDHG_OK;
  for (int l = 0; l < count; ++l) {
    ResLp& p = d->lps[l];
    p.C = Cs[l];
    p.own_m = res_own(p.m, p.C);
    p.own_n = res_own(p.n, p.C);
  }
  const std::vector<int32_t> list = res_order(d->lps, ops);
  d->groups.clear();
  for (int i = 0; i < count; ++i) {
    const ResLp& p = d->lps[list[i]];
    if (d->groups.empty() || d->groups.back().C != p.C) d->groups.push_back(ResGroup{p.C, i, 0});
    ResGroup& g = d->groups.back();
    g.count += 1;
    g.smem_solve = std::max(g.smem_solve, cg_smem(p.m, p.n, p.C));
  }
  for (const ResGroup& g : d->groups)
    if (!res_fits(cg_kernel(g.C), g.C, g.smem_solve, ctx->smem_optin)) return PDHG_OK;
  CK(d->side.make((int)d->groups.size()));
  if (!d->lp) {
    // slices pad a matrix by less than 0.3 of its entries plus 2048 per LP
    // (rows sorted by length: a lane's row is at most the slice before's
    // shortest; 8 and 32 lanes round rows above 24 and 256 up to a step)
    d->cap = (size_t)(ctx->nnz + ctx->nnz / 10 * 3) + 2048 * (size_t)count;
    const size_t z = (size_t)ctx->nnz;
    CKS(dalloc(ctx, &d->list, (size_t)count));
    CKS(dalloc(ctx, &d->a_sl, (size_t)m));
    CKS(dalloc(ctx, &d->t_sl, (size_t)n));
    CKS(dalloc(ctx, &d->ord_m, (size_t)m));
    CKS(dalloc(ctx, &d->ord_n, (size_t)n));
    CKS(dalloc(ctx, &d->pos_m, (size_t)m));
    CKS(dalloc(ctx, &d->pos_n, (size_t)n));
    CKS(dalloc(ctx, &d->a_col, d->cap));
    CKS(dalloc(ctx, &d->t_col, d->cap));
    for (int o = 0; o < 2; ++o)
      for (int k = 0; k < 2; ++k) CKS(dalloc(ctx, &d->val[o][k], d->cap));
    CKS(dalloc(ctx, &d->idx, (size_t)n + 1));
    CKS(dalloc(ctx, &d->bcol, (size_t)n));
    CKS(dalloc(ctx, &d->len, (size_t)std::max(m, n)));
    CKS(dalloc(ctx, &d->scan, (size_t)std::max(m, n) / 1024 + 8));
    CKS(dalloc(ctx, &d->sa_rp, (size_t)m + 1));
    CKS(dalloc(ctx, &d->st_rp, (size_t)n + 1));
    CKS(dalloc(ctx, &d->sa_col, std::max(z, (size_t)m)));
    CKS(dalloc(ctx, &d->sa_src, z));
    CKS(dalloc(ctx, &d->st_col, z));
    CKS(dalloc(ctx, &d->st_src, z));
    CKS(dalloc(ctx, &d->iters, (size_t)count));
    CKS(dalloc(ctx, &d->flags, 2));
    CKS(dalloc(ctx, &d->elems, 2 * (size_t)count));
    CKS(dalloc(ctx, &d->lp, (size_t)count));
  }
  cudaStream_t s = ctx->stream;
  const int gn = std::max(1, std::min((n + 255) / 256, ctx->nsm * 8));
  const int gm = std::max(1, std::min((std::max(n, 8 * m) + 255) / 256, ctx->nsm * 8));
  CK(cudaMemcpyAsync(d->lp, d->lps.data(), sizeof(ResLp) * count, cudaMemcpyHostToDevice, s));
  CK(cudaMemcpyAsync(d->list, list.data(), sizeof(int32_t) * count, cudaMemcpyHostToDevice, s));
  CK(cudaMemsetAsync(d->flags, 0, 2 * sizeof(int32_t), s));
  k_sub_flags<<<gn, 256, 0, s>>>(n, mask, d->len);
  launch_scan(d->len, d->idx, n, d->scan, s);
  int32_t* a_len = d->sa_col;  // counted here first, scanned, then overwritten
  k_sub_count<<<gm, 256, 0, s>>>(m, n, ctx->a_rp, ctx->a_col, ctx->t_rp, mask, d->idx, d->bcol, d->len,
                                 a_len);
  launch_scan(a_len, d->sa_rp, m, d->scan, s);
  launch_scan(d->len, d->st_rp, (int)nb, d->scan, s);
  k_sub_fill<<<gm, 256, 0, s>>>(m, (int)nb, ctx->a_rp, ctx->a_col, ctx->t_rp, ctx->t_col, mask, d->idx,
                                d->bcol, d->sa_rp, d->st_rp, d->sa_col, d->sa_src, d->st_col, d->st_src);
  launch_res_sort(ResBuild{d->lp, d->sa_rp, d->st_rp, d->a_sl, d->t_sl, d->ord_m, d->ord_n, d->pos_m,
                           d->pos_n, d->elems, d->flags},
                  count, s);
  ctx->launches += 13;
  std::vector<long long> el(2 * (size_t)count);
  CK(cudaMemcpyAsync(el.data(), d->elems, sizeof(long long) * el.size(), cudaMemcpyDeviceToHost, s));
  CK(cudaMemcpyAsync(d->lps.data(), d->lp, sizeof(ResLp) * count, cudaMemcpyDeviceToHost, s));
  CK(cudaStreamSynchronize(s));
  int64_t ea = 0, et = 0;
  d->max_slices = 1;
  for (int l = 0; l < count; ++l) {
    d->lps[l].a_el = ea;
    d->lps[l].t_el = et;
    ea += el[2 * l];
    et += el[2 * l + 1];
    d->max_slices = std::max({d->max_slices, d->lps[l].a_slices, d->lps[l].t_slices});
  }
  if ((size_t)std::max(ea, et) > d->cap) return PDHG_OK;  // never above the bound; the tile kernels remain
  CK(cudaMemcpyAsync(d->lp, d->lps.data(), sizeof(ResLp) * count, cudaMemcpyHostToDevice, s));
  CK(cudaStreamSynchronize(s));
  d->ready = true;
  return PDHG_OK;
}

pdhg_status resident_cg_layout(pdhg_ctx* ctx, ResCgData* d, const double* mask, const int32_t* active) {
  const bool had = d->lp != nullptr;  // (the arrays are kept between layouts)
  return if_room(ctx, [&] { return cg_layout(ctx, d, mask, active); },
                 [&] {
                   d->ready = false;
                   if (!had) d->lp = nullptr;
                 });
}

// w (start in, solution out) of M_B^T M_B w = rhs per LP, M the scaled matrix
// (original = false) or the given one
pdhg_status resident_cg(pdhg_ctx* ctx, ResCgData* d, bool original, const double* rhs, double* w,
                        double tol, int max_iter, std::vector<int32_t>* iters) {
  const int count = ctx->count, o = original ? 1 : 0;
  cudaStream_t s = ctx->stream;
  if (!original || !d->original) {  // the scaled ones come first and bring the columns
    launch_res_fill(ResFill{d->lp, d->sa_rp, d->st_rp, d->sa_col, d->st_col,
                            original ? ctx->a_val_orig : ctx->a_val64,
                            original ? ctx->t_val_orig : ctx->t_val64, d->sa_src, d->st_src, d->a_sl,
                            d->t_sl, d->ord_m, d->ord_n, d->pos_m, d->pos_n,
                            original ? nullptr : d->a_col, original ? nullptr : d->t_col, d->val[o][0],
                            d->val[o][1], nullptr, nullptr},
                    count, d->max_slices, s);
    ctx->launches += 1;
    if (original) d->original = true;
  }
  ResCg A{d->lp,   nullptr, d->a_sl,      d->t_sl,      d->a_col, d->t_col, d->ord_n,
          d->val[o][0], d->val[o][1], d->bcol, rhs, w, d->iters, tol * tol, max_iter,
          (unsigned long long)ctx->opt.wait_limit_ms * 1000000ull, res_tx_extra(ctx), d->flags + 1};
  CK(cudaMemsetAsync(d->flags + 1, 0, sizeof(int32_t), s));
  CKS(res_groups(ctx, d->groups, d->side, [&](const ResGroup& g, cudaStream_t q) {
    A.list = d->list + g.first;
    cudaLaunchAttribute attr;
    const cudaLaunchConfig_t cfg = res_config(g.C, g.count, g.smem_solve, q, &attr);
    cudaError_t e = cudaSuccess;
    RES_DISPATCH_C(g.C, e = cudaLaunchKernelEx(&cfg, k_res_cg<C_>, A));
    return e;
  }));
  int32_t err = 0;
  iters->resize((size_t)count);
  CK(cudaMemcpyAsync(&err, d->flags + 1, sizeof(err), cudaMemcpyDeviceToHost, s));
  CK(cudaMemcpyAsync(iters->data(), d->iters, sizeof(int32_t) * count, cudaMemcpyDeviceToHost, s));
  CK(cudaStreamSynchronize(s));
  if (err) {
    set_error("conjugate gradients: a CTA waited longer than options.wait_limit_ms for another's vector");
    return PDHG_TIMEOUT;
  }
  return PDHG_OK;
}

}  // namespace pdhg
