// The solve of LPs that fit on chip (resident.cuh): the kernel and its launch,
// instantiated per precision in resident_f32.cu and resident_f64.cu.
#pragma once
#include "dispatch.cuh"
#include "eval_rule.cuh"
#include "kernels.h"
#include "resident.cuh"

namespace pdhg {

// One cluster per LP, from its stored state until it has finished or slice_ns
// has passed (the state is stored exactly, so where a launch ends changes
// nothing).  Bound by the float64 pipe in float64 (2 operations per clock and
// SM: 512 LPs of 50..5000 rows to 1e-4 in 38.5 ms against 126 ms of the tile
// kernels' launches, about 0.9 of that pipe while every SM has an LP), by the
// latency of one pass over a slice and of two exchanges per iteration where an
// LP has the chip to itself (2000 x 5000 float64 3.7 us per iteration against
// 11.4, 97 LPs float32-mixed 192 iterations in 1.9 ms against 4.8).  512 threads
// of up to 128 registers: two CTAs per SM at 64 registers spilled and were 5 to
// 30% slower.
template <typename T, int C, bool hal>
__global__ void __launch_bounds__(kResThreads) k_res_solve(ResSolve<T> A) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ double tot[16];
  const int l = A.list[blockIdx.x / C];
  const ResLp lp = A.lp[l];
  const ResSmem L = res_smem(lp.m, lp.n, lp.own_m, lp.own_n, hal ? 6 : 4, hal ? 4 : 2, sizeof(T));
  const ResCluster<C> cl(smem);
  const IterBuffers<T>& B = A.B;
  Scalars& sc = *reinterpret_cast<Scalars*>(smem + L.sc);
  T* X = reinterpret_cast<T*>(smem + L.X);
  T* Y = reinterpret_cast<T*>(smem + L.Y);
  T* tab = reinterpret_cast<T*>(smem + L.tab);
  // the CTA's own columns and rows (slots of its slices)
  T* xa = reinterpret_cast<T*>(smem + L.own_n);
  T* cc = xa + lp.own_n;
  T* xo = cc + lp.own_n;   // Halpern: z's x (X holds T(z)'s) and the anchor
  T* x0 = xo + lp.own_n;
  T* ya = reinterpret_cast<T*>(smem + L.own_m);
  T* ax = ya + lp.own_m;
  T* axa = ax + lp.own_m;
  T* bb = axa + lp.own_m;
  T* y0 = bb + lp.own_m;
  T* ax0 = y0 + lp.own_m;
  const int tid = threadIdx.x;
  const unsigned long long t0 = global_ns();
  if (tid == 0) sc = B.sc[l];
  __syncthreads();
  const bool was_done = sc.done != 0;  // the same on every CTA of the cluster
  if (was_done) return;
  const ResMat Mt(A.t_sl + lp.n_off, A.t_col + lp.t_el, lp.t_slices, cl.rank, C);
  const ResMat Ma(A.a_sl + lp.m_off, A.a_col + lp.a_el, lp.a_slices, cl.rank, C);
  const T* tv = A.t_val + lp.t_el;
  const T* av = A.a_val + lp.a_el;
  const uint16_t* on = A.ord_n + lp.n_off;
  const uint16_t* om = A.ord_m + lp.m_off;
  // X and Y of an iteration travel by transaction-counted stores
  const uint32_t bar_x = L.bar, bar_y = L.bar + 8u;
  const uint32_t bytes_x = (uint32_t)(lp.n * sizeof(T)) + A.tx_extra,
                 bytes_y = (uint32_t)(lp.m * sizeof(T)) + A.tx_extra;
  uint32_t phase = 0;  // the parity of both barriers' current phase
  const bool idle = C > 1 && res_idle(Ma, Mt);
  if (C > 1 && tid == 0) {
    mbar_init(cl.base + bar_x);
    mbar_init(cl.base + bar_y);
    mbar_arrive_expect(cl.base + bar_x, bytes_x);
    mbar_arrive_expect(cl.base + bar_y, bytes_y);
  }
  if (tid < kResMaxC) reinterpret_cast<double*>(smem + L.rec)[tid * 18 + 17] = 0.0;
  bool lost = false;  // a wait ran out (uniform in a warp, which sends nothing more)
  auto push_x = [&](int p, T v) { cl.push(L.X + (uint32_t)p * (uint32_t)sizeof(T), v); };
  auto push_y = [&](int p, T v) { cl.push(L.Y + (uint32_t)p * (uint32_t)sizeof(T), v); };
  cl.sync();  // every CTA of the cluster has started (its shared memory may be written)
  Mt.template each<C>([&](const ResSlice& s, int row) {
    if (row < 0) return;
    const int p = s.p0 + row, k = s.loc + row;
    const int64_t j = lp.n_off + on[p];
    xa[k] = B.x_avg[j];
    cc[k] = B.c_t[j];
    if (hal) {
      xo[k] = B.x[j];
      x0[k] = B.x_last[j];
      push_x(p, xa[k]);
    } else {
      push_x(p, B.x[j]);
    }
  });
  Ma.template each<C>([&](const ResSlice& s, int row) {
    if (row < 0) return;
    const int p = s.p0 + row, k = s.loc + row;
    const int64_t i = lp.m_off + om[p];
    ya[k] = B.y_avg[i];
    ax[k] = B.Ax[i];
    axa[k] = B.Ax_avg[i];
    bb[k] = B.b_t[i];
    if (hal) {
      y0[k] = B.y_last[i];
      ax0[k] = B.Ax_last[i];
    }
    push_y(p, B.y[i]);
  });
  if (tid == 0) {
    X[lp.n] = T(0);
    Y[lp.m] = T(0);
  }
  cl.sync();
  const T rho = (T)B.rho;
  bool stop = false;
  while (!stop) {
    const long long k0 = sc.k, F = sc.eval_freq, tt0 = sc.t;
    const long long next = min((k0 / F + 1) * F, sc.max_iter);
    const int len = (int)(next - k0);
    const T tau = (T)sc.tau, sigma = (T)sc.sigma;
    const uint32_t phase0 = phase;
    int sent = 0, seen = 0;  // half-steps of this chunk that the warp has computed, seen arrive
    for (int i = 0; i < len; ++i) {
      if ((i & 63) == 0) {
        // The next 64 weights (a float64 division each), by warp 0: it has seen
        // the last Y complete, so every warp with rows has taken its last weight;
        // a warp without rows may be here while the others still read the table.
        if (tid < 32) {
#pragma unroll
          for (int e = tid; e < 64; e += 32) {
            const long long tt = tt0 + i + e;
            tab[e] = hal ? halpern_weight(tt + 1, T(0)) : avg_weight(tt + 1, T(0));
          }
        }
        lost = __syncthreads_or(lost);
        if (lost) break;
      }
      const T w = tab[i & 63];
      const bool first = tt0 + i == 0;
      if (C == 1 || !lost) Mt.template each<C>([&](const ResSlice& s, int row) {
        const T* const buf[1] = {Y};
        const int p = s.p0 + row, k = s.loc + row;
        T d[1] = {row >= 0 ? cc[k] : T(0)};  // c~ - A~^T y, the sum starting at c~
        const T x = row >= 0 ? (hal ? xo[k] : X[p]) : T(0);
        res_dot<1, true>(s, tv, Mt.col, buf, d);
        if (row < 0) return;
        const T xn = max0(x - tau * d[0]);
        cl.send(L.X + (uint32_t)p * (uint32_t)sizeof(T), bar_x, xn);
        if (hal) {
          xa[k] = xn;
          xo[k] = w * ((T(1) + rho) * xn - rho * x) + (T(1) - w) * x0[k];
        } else {
          const T a = xa[k];
          xa[k] = first ? xn : a + (xn - a) * w;
        }
      });
      sent += !lost;
      if constexpr (C == 1) cl.sync();
      else if (!lost && !idle) lost = !cl.arrived(bar_x, phase, bytes_x, A.wait_ns);
      seen += !lost;
      if (C == 1 || !lost) Ma.template each<C>([&](const ResSlice& s, int row) {
        const T* const buf[1] = {X};
        T h1[1] = {T(0)};
        res_dot<1, false>(s, av, Ma.col, buf, h1);
        if (row < 0) return;
        const int p = s.p0 + row, k = s.loc + row;
        const T h = h1[0], y = Y[p], axo = ax[k];
        const T yh = y + sigma * (bb[k] - (h + h) + axo);
        const T yn = hal ? w * ((T(1) + rho) * yh - rho * y) + (T(1) - w) * y0[k] : yh;
        cl.send(L.Y + (uint32_t)p * (uint32_t)sizeof(T), bar_y, yn);
        if (hal) {
          ya[k] = yh;
          axa[k] = h;
          ax[k] = w * ((T(1) + rho) * h - rho * axo) + (T(1) - w) * ax0[k];
        } else {
          const T a = ya[k], b = axa[k];
          ax[k] = h;
          ya[k] = first ? yn : a + (yn - a) * w;
          axa[k] = first ? h : b + (h - b) * w;
        }
      });
      sent += !lost;
      if constexpr (C == 1) cl.sync();
      else if (!lost && !idle) lost = !cl.arrived(bar_y, phase, bytes_y, A.wait_ns);
      seen += !lost;
      phase ^= 1u;
    }
    // a wait that ran out: tell every CTA (each comes to the next cluster
    // barrier, since all its waits are bounded)
    if constexpr (C > 1) {
      if (__syncthreads_or(lost) && tid == 0) cl.push(L.rec + (uint32_t)(cl.rank * 18 + 17) * 8u, 1.0);
    }
    // evaluation: x and y go to their natural places (they come back below),
    // the copies of x make room for the average of y
    Mt.template each<C>([&](const ResSlice& s, int row) {
      if (row >= 0) B.x[lp.n_off + on[s.p0 + row]] = hal ? xo[s.loc + row] : X[s.p0 + row];
    });
    Ma.template each<C>([&](const ResSlice& s, int row) {
      if (row >= 0) B.y[lp.m_off + om[s.p0 + row]] = Y[s.p0 + row];
    });
    cl.sync();
    if constexpr (C > 1) {
      bool any = false;
#pragma unroll
      for (int q = 0; q < C; ++q) any |= reinterpret_cast<const double*>(smem + L.rec)[q * 18 + 17] != 0.0;
      if (any) {  // the whole cluster leaves, each CTA when what was sent to it has arrived
        if (tid == 0) atomicExch(A.err, 1);
        double n[2] = {0.0, 0.0};
        Mt.template each<C>([&](const ResSlice&, int row) { n[0] += row >= 0; });
        Ma.template each<C>([&](const ResSlice&, int row) { n[1] += row >= 0; });
        n[0] *= (sent + 1) / 2;
        n[1] *= sent / 2;
        res_reduce<2>(cl, L, smem, n, tot);
        if (tid == 0) {
          const int x = (seen + 1) / 2, y = seen / 2;
          cl.drain(bar_x, phase0 ^ (x & 1), (long long)tot[0] * sizeof(T), (1ll + x) * bytes_x, A.wait_ns);
          cl.drain(bar_y, phase0 ^ (y & 1), (long long)tot[1] * sizeof(T), (1ll + y) * bytes_y, A.wait_ns);
        }
        return;
      }
    }
    Ma.template each<C>([&](const ResSlice& s, int row) {
      if (row >= 0) push_x(s.p0 + row, ya[s.loc + row]);
    });
    if (tid == 0) X[lp.m] = T(0);
    cl.sync();
    double q[16];
#pragma unroll
    for (int e = 0; e < 16; ++e) q[e] = 0.0;
    Mt.template each<C>([&](const ResSlice& s, int row) {
      const T* const buf[2] = {Y, X};
      T g[2] = {T(0), T(0)};
      res_dot<2, false>(s, tv, Mt.col, buf, g);
      if (row < 0) return;
      const int64_t j = lp.n_off + on[s.p0 + row];
      const double cj = B.c_t64[j], dci = B.Dc_inv[j], xl = (double)B.x_last[j];
      const double xs[2] = {(double)B.x[j], (double)xa[s.loc + row]};
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const double rd = min0(cj - (double)g[e]), ru = rd * dci, dx = xs[e] - xl;
        q[e * Q_N + Q_S2] += rd * rd;
        q[e * Q_N + Q_U2] += ru * ru;
        q[e * Q_N + Q_S3] += cj * xs[e];
        q[e * Q_N + Q_D1] += dx * dx;
      }
    });
    Ma.template each<C>([&](const ResSlice& s, int row) {
      if (row < 0) return;
      const int k = s.loc + row;
      const int64_t i = lp.m_off + om[s.p0 + row];
      const double bi = B.b_t64[i], dri = B.Dr_inv[i], yl = (double)B.y_last[i];
      const double axs[2] = {(double)ax[k], (double)axa[k]};
      const double ys[2] = {(double)Y[s.p0 + row], (double)ya[k]};
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const double rp = bi - axs[e], ru = rp * dri, dy = ys[e] - yl;
        q[e * Q_N + Q_S1] += rp * rp;
        q[e * Q_N + Q_U1] += ru * ru;
        q[e * Q_N + Q_S4] += bi * ys[e];
        q[e * Q_N + Q_D2] += dy * dy;
      }
    });
    const bool late = res_reduce<16>(cl, L, smem, q, tot, tid == 0 && global_ns() - t0 > A.slice_ns);
    // every CTA applies the rule to its own copy of the scalars (the same
    // sums, the same decision); rank 0 keeps the log
    if (tid < 32) {
      const EvalRoots R = eval_roots_warp(sc, tot);
      if (tid == 0)
        apply_eval_rule(sc, tot, len, R, cl.rank == 0 ? B.log_k : nullptr, B.log_flags, B.log_kkt);
    }
    __syncthreads();
    if constexpr (sizeof(T) == 4) {
      if (sc.verify) {
        // float64 check of the candidate that passed the screen
        const bool avg = sc.verify_avg != 0;
        cl.sync();
        Mt.template each<C>([&](const ResSlice& s, int row) {
          if (row >= 0) push_x(s.p0 + row, avg ? xa[s.loc + row] : B.x[lp.n_off + on[s.p0 + row]]);
        });
        Ma.template each<C>([&](const ResSlice& s, int row) {
          if (row >= 0) push_y(s.p0 + row, avg ? ya[s.loc + row] : B.y[lp.m_off + om[s.p0 + row]]);
        });
        if (tid == 0) X[lp.n] = T(0);
        cl.sync();
        double r[4] = {0.0, 0.0, 0.0, 0.0};
        Mt.template each<C>([&](const ResSlice& s, int row) {
          const T* const buf[1] = {Y};
          double g[1] = {0.0};
          res_dot<1, false>(s, A.t_val64 + lp.t_el, Mt.col, buf, g);
          if (row < 0) return;
          const int64_t j = lp.n_off + on[s.p0 + row];
          const double cj = B.c_t64[j], rd = min0(cj - g[0]) * B.Dc_inv[j];
          r[0] += rd * rd;
          r[1] += cj * (double)X[s.p0 + row];
        });
        Ma.template each<C>([&](const ResSlice& s, int row) {
          const T* const buf[1] = {X};
          double h[1] = {0.0};
          res_dot<1, false>(s, A.a_val64 + lp.a_el, Ma.col, buf, h);
          if (row < 0) return;
          const int64_t i = lp.m_off + om[s.p0 + row];
          const double bi = B.b_t64[i], rp = (bi - h[0]) * B.Dr_inv[i];
          r[2] += rp * rp;
          r[3] += bi * (double)Y[s.p0 + row];
        });
        res_reduce<4>(cl, L, smem, r, tot);
        if (tid == 0) {
          const bool log = cl.rank == 0;
          eval_fp64_check(sc, tot[2], tot[0], tot[1], tot[3], log ? B.log_k : nullptr, B.log_flags,
                          B.log_kkt);
        }
        __syncthreads();
      }
    }
    stop = sc.done != 0 || late;
    // the restart, and the iterate back into the copies
    const bool re = sc.restart_pending != 0, to_avg = re && sc.restart_to_avg != 0;
    cl.sync();
    Mt.template each<C>([&](const ResSlice& s, int row) {
      if (row < 0) return;
      const int p = s.p0 + row, k = s.loc + row;
      const int64_t j = lp.n_off + on[p];
      const T x = to_avg ? xa[k] : B.x[j];
      if (to_avg) B.x[j] = x;
      if (re) B.x_last[j] = x;
      if (hal) {
        xo[k] = x;
        if (re) x0[k] = x;
        push_x(p, xa[k]);
      } else {
        push_x(p, x);
      }
    });
    Ma.template each<C>([&](const ResSlice& s, int row) {
      if (row < 0) return;
      const int p = s.p0 + row, k = s.loc + row;
      const int64_t i = lp.m_off + om[p];
      const T y = to_avg ? ya[k] : B.y[i];
      if (to_avg) {
        B.y[i] = y;
        ax[k] = axa[k];
      }
      if (re) {
        B.y_last[i] = y;
        B.Ax_last[i] = ax[k];
        if (hal) {
          y0[k] = y;
          ax0[k] = ax[k];
        }
      }
      push_y(p, y);
    });
    __syncthreads();
    if (tid == 0) {
      X[lp.n] = T(0);
      sc.restart_pending = 0;
    }
    cl.sync();
  }
  Mt.template each<C>([&](const ResSlice& s, int row) {
    if (row >= 0) B.x_avg[lp.n_off + on[s.p0 + row]] = xa[s.loc + row];
  });
  Ma.template each<C>([&](const ResSlice& s, int row) {
    if (row < 0) return;
    const int k = s.loc + row;
    const int64_t i = lp.m_off + om[s.p0 + row];
    B.y_avg[i] = ya[k];
    B.Ax[i] = ax[k];
    B.Ax_avg[i] = axa[k];
  });
  if (cl.rank == 0 && tid == 0) {
    B.sc[l] = sc;
    if (sc.done) atomicSub(A.active, 1);
  }
}


// the kernel for clusters of C CTAs
template <typename T>
const void* res_solve_kernel(int C, bool halpern) {
  constexpr bool H = sizeof(T) == 8;  // float32 runs in batches, which have no Halpern form
  const void* f = nullptr;
  RES_DISPATCH_C(C, f = halpern ? (const void*)k_res_solve<T, C_, H>
                                : (const void*)k_res_solve<T, C_, false>);
  return f;
}
template <typename T>
cudaError_t launch_res_solve(const ResSolve<T>& A, int C, int lps, size_t smem, bool halpern,
                             cudaStream_t s) {
  constexpr bool H = sizeof(T) == 8;
  cudaLaunchAttribute attr;
  const cudaLaunchConfig_t cfg = res_config(C, lps, smem, s, &attr);
  cudaError_t e = cudaSuccess;
  RES_DISPATCH_C(C, e = halpern ? cudaLaunchKernelEx(&cfg, k_res_solve<T, C_, H>, A)
                                : cudaLaunchKernelEx(&cfg, k_res_solve<T, C_, false>, A));
  return e;
}

}  // namespace pdhg
