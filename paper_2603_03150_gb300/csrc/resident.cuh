// On-chip LPs: one thread-block cluster holds an LP's iterate in shared memory
// for a whole solve (the layout, its build and the device helpers shared by
// the solve, the power iteration and the conjugate gradients).
//
// Layout.  Each matrix of an LP (A~ and A~^T) is stored in slices of one warp:
// the rows are sorted by length (longest first, stable, so the order is
// fixed), rows of up to kResShort nonzeros go 32 to a slice (a lane each; 16 or 8
// in small LPs), rows of up to kResMid 4 to a slice (8 lanes each), longer ones one to a
// slice.  Step k of a slice is 32 consecutive values and 16-bit columns, so
// the loads coalesce and a row costs one fused multiply-add per nonzero and,
// for the longer classes, the shuffle sum: GB300 runs 2 float64 operations per
// clock and SM, so the segmented scan of the CSR tiles (5 float64 additions
// for 8 nonzeros) is what this layout leaves out.  Columns are positions in
// the sorted order of the other matrix, in which the vectors are kept too.
// Entries past a row's end have value 0 and the column of a slot that holds 0.
//
// Slice s belongs to CTA s mod C of the cluster and warp (s / C) mod kResWarps
// of it: always the same lane works on a row, so the row's own operands need
// no barrier.  Every CTA holds the whole gathered vectors; a new entry is
// written to all C copies through distributed shared memory.
//
// Who waits.  A half-step ends for a warp when its CTA's transaction barrier has
// counted the whole vector.  The wait names a phase by its parity alone, so a
// warp must have seen a phase before the next one completes.  Two things hold a
// warp to that: it has rows (the vector after next cannot be complete without
// them, and it computes them behind the wait), or it is warp 0, whose thread
// arms the barrier's next phase.  A warp without a slice of either matrix has
// neither: the LP 200 x 500 leaves 12 of a CTA's 16 warps in that state, and one
// that was a whole iteration late would have taken a phase that is over for one
// that never ends.  It reads no vector, so it does not wait for them: the block
// barriers that all warps meet (every 64 iterations and at an evaluation in the
// solve, in every sum of the power iteration and the conjugate gradients) hold it.
#pragma once
#include "common.cuh"
#include "kernels.h"

namespace pdhg {

constexpr int kResThreads = 512, kResWarps = kResThreads / 32;
constexpr int kResShort = 24;   // a lane per row up to this many nonzeros
constexpr int kResMid = 256;    // 8 lanes per row up to this many, a warp above
constexpr int kResMaxC = 16;    // CTAs of a cluster (16 needs the non-portable size)
// What is solved on chip, and by how many CTAs (us per iteration, one LP, GB300,
// one lane per short row; tile kernels: 10 at 200 x 500, 11.4 at 2000 x 5000):
//   float64, clusters of 1 / 4 / 16: 60 x 150 2.4 / 2.6 / 2.7, 200 x 500 3.4 /
//   2.5 / 2.7, 2000 x 5000 23.7 / 7.1 / 3.7; float32: 1.1 / 1.3 / 1.5, 1.4 / 1.4
//   / 1.5, 9.8 / 3.1 / 2.3.
// So a CTA gets at least kResMinOps operations of an iteration (an exchange
// between CTAs costs about 250 clocks).  Above kResMaxNnz nonzeros 16 CTAs do
// not outrun the whole chip's tile kernels, and a row longer than kResMaxRow
// would be a chain of more than 128 steps in one warp.
constexpr int64_t kResMaxNnz = 320000;
constexpr int kResMaxRow = 4096;
constexpr double kResMinOps64 = 3000.0, kResMinOps32 = 6000.0;

struct ResSlice {
  int32_t off;  // first element of the slice, relative to the LP's matrix
  int32_t p0;   // position of its first row
  int32_t loc;  // slot of its first row among its CTA's own rows
  int32_t wgr;  // steps | log2(lanes per row) << 16 | rows << 20
};
__host__ __device__ constexpr int res_steps(int wgr) { return wgr & 0xffff; }
__host__ __device__ constexpr int res_lg(int wgr) { return (wgr >> 16) & 15; }
__host__ __device__ constexpr int res_rows(int wgr) { return wgr >> 20; }

struct ResLp {
  int32_t m, n;
  int64_t m_off, n_off;  // its first row / column in the stacked arrays (and first slice)
  int64_t a_el, t_el;    // first element of its slices of A~ / A~^T
  int32_t C;             // CTAs of its cluster
  int32_t a_slices, t_slices;
  int32_t own_m, own_n;  // slots of a CTA's own rows and columns (bounds)
  int32_t lg_a, lg_t;    // log2 of the lanes of a short row of A~ / A~^T
};

// Lanes (log2) of a short row of a matrix whose slices are few: an iteration then
// waits for the chains of dependent additions (68 clocks each), not for the
// float64 pipe (a warp's operation takes 16 clocks of it).  Twice the lanes while
// a CTA has less than 3 slices (it has less than 6 after) and a lane 6 nonzeros.
// us per iteration with 1 / 2 / 4 lanes for the rows of A~ (12.5 nonzeros),
// float64: 30 x 80 2.18 / 1.79 / 1.64, 60 x 150 2.38 / 1.94 / 2.11, 200 x 500
// 2.55 / 2.14 / 2.16, 2000 x 5000 3.94 / 4.24 / 5.02; 2 lanes for the rows of
// A~^T (5 nonzeros) 200 x 500 2.14 -> 2.20.
__host__ inline int res_lanes(int rows, int64_t nnz, int C) {
  int lg = 0;
  while (lg < 2 && ((int64_t)rows << lg) <= 90LL * C && nnz >= ((int64_t)rows * 6 << lg)) ++lg;
  return lg;
}

// Slots of one CTA's own rows of a matrix of `rows` rows: a class of slices
// dealt to C CTAs gives a CTA at most one slice above the mean.
__host__ __device__ inline int res_own(int rows, int C) { return rows / C + 73; }

// Dynamic shared memory of a cluster's CTA.  own_n / own_m: T vectors of the
// CTA's own columns / rows (nvn, nvm of them); X and Y the gathered copies.
struct ResSmem {
  uint32_t sc, rec, red, tab, bar, X, Y, own_n, own_m, total;
};
__host__ __device__ inline ResSmem res_smem(int m, int n, int own_m, int own_n, int nvm, int nvn,
                                            int es) {
  ResSmem r;
  uint32_t o = 0;
  auto take = [&](uint32_t bytes) {
    const uint32_t at = o;
    o = (o + bytes + 15u) & ~15u;
    return at;
  };
  r.sc = take(sizeof(Scalars));
  r.rec = take(kResMaxC * 18 * 8);   // one record per CTA: 16 sums, 2 flags
  r.red = take(nvm ? 16 * kResWarps * 8 : (2 * kResThreads + 8) * 8);  // (no vectors of rows: ResExchange)
  r.tab = take(64 * 8);              // averaging weights of 64 iterations
  r.bar = take(32);                  // transaction barriers: X, Y and two sums
  r.X = take((uint32_t)(((m > n ? m : n) + 1) * es));
  r.Y = take((uint32_t)((m + 1) * es));
  r.own_n = take((uint32_t)(own_n * nvn * es));
  r.own_m = take((uint32_t)(own_m * nvm * es));
  r.total = o;
  return r;
}

// A cluster of C CTAs, one of its CTAs (rank) with its shared memory window.
template <int C>
struct ResCluster {
  uint32_t base;  // this CTA's dynamic shared memory
  int rank;
  __device__ __forceinline__ ResCluster(void* smem) {
    base = (uint32_t)__cvta_generic_to_shared(smem);
    rank = 0;
    if constexpr (C > 1) {
      uint32_t r;
      asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
      rank = (int)r;
    }
  }
  // offset `off` of rank q's dynamic shared memory
  __device__ __forceinline__ uint32_t at(int q, uint32_t off) const {
    uint32_t a;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(base + off), "r"(q));
    return a;
  }
  // all threads of all CTAs; what was pushed before is visible after
  __device__ __forceinline__ void sync() const {
    if constexpr (C == 1) {
      __syncthreads();
    } else {
      asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
      asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    }
  }
  // v to offset off on every CTA, visible after the next sync()
  __device__ __forceinline__ void push(uint32_t off, double v) const {
    if constexpr (C == 1)
      asm volatile("st.shared.f64 [%0], %1;" ::"r"(base + off), "d"(v) : "memory");
    else
#pragma unroll 2
      for (int q = 0; q < C; ++q)
        asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(at(q, off)), "d"(v) : "memory");
  }
  __device__ __forceinline__ void push(uint32_t off, float v) const {
    if constexpr (C == 1)
      asm volatile("st.shared.f32 [%0], %1;" ::"r"(base + off), "f"(v) : "memory");
    else
#pragma unroll 2
      for (int q = 0; q < C; ++q)
        asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(at(q, off)), "f"(v) : "memory");
  }
  // v to offset off on every CTA, counted by the transaction barrier at offset
  // bar of each: a CTA that has seen a whole vector arrive knows that every
  // row of the half-step has been computed, so no other barrier is needed
  // (C = 1: plain stores, the caller meets sync())
  __device__ __forceinline__ void send(uint32_t off, uint32_t bar, double v) const {
    if constexpr (C == 1) {
      push(off, v);
    } else {
#pragma unroll 4
      for (int q = 0; q < C; ++q)
        asm volatile(
            "st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.b64 [%0], %1, [%2];" ::"r"(at(q, off)),
            "l"(__double_as_longlong(v)), "r"(at(q, bar))
            : "memory");
    }
  }
  __device__ __forceinline__ void send(uint32_t off, uint32_t bar, float v) const {
    if constexpr (C == 1) {
      push(off, v);
    } else {
#pragma unroll 4
      for (int q = 0; q < C; ++q)
        asm volatile(
            "st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.b32 [%0], %1, [%2];" ::"r"(at(q, off)),
            "r"(__float_as_int(v)), "r"(at(q, bar))
            : "memory");
    }
  }
  __device__ __forceinline__ void send_to(int q, uint32_t off, uint32_t bar, double v) const {
    if constexpr (C == 1)
      push(off, v);
    else
      asm volatile(
          "st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.b64 [%0], %1, [%2];" ::"r"(at(q, off)),
          "l"(__double_as_longlong(v)), "r"(at(q, bar))
          : "memory");
  }
  // waits until the vector counted by barrier `bar` has arrived (phase parity)
  // and lets thread 0 expect the next one; false (for the whole warp) once a
  // lane's wait ran past limit_ns.  Only for warps that cannot miss a phase (see
  // the head of this file).
  __device__ __forceinline__ bool arrived(uint32_t bar, uint32_t parity, uint32_t bytes,
                                          unsigned long long limit_ns) const {
    const uint32_t mb = base + bar;
    unsigned long long t0 = 0;
    uint32_t done = 0;
    for (uint32_t n = 0; !done; ++n) {
      asm volatile(
          "{ .reg .pred p; mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2; "
          "selp.u32 %0, 1, 0, p; }"
          : "=r"(done)
          : "r"(mb), "r"(parity)
          : "memory");
      if ((n & 255u) == 255u) {
        if (t0 == 0) t0 = global_ns();
        else if (global_ns() - t0 > limit_ns) break;
      }
    }
    const bool ok = __all_sync(0xffffffffu, done != 0);
    if (threadIdx.x == 0 && ok) mbar_arrive_expect(mb, bytes);
    return ok;
  }
  // Thread 0, on its way out after a wait that ran out: waits until everything
  // that was sent to this CTA over barrier `bar` has arrived.  A CTA must not
  // exit while a store is on its way to it, and neither a cluster barrier nor a
  // delay tells that none is.  The barrier counts bytes: thread 0 has let it
  // expect `armed` so far (the last phase, of the given parity, is the one that
  // is open), and all CTAs together have sent `sent`.  What was expected and
  // not sent is counted as arrived; what was sent beyond it (a CTA may be one
  // exchange ahead) is a phase of its own.  Bounded by limit_ns a phase.
  __device__ __forceinline__ void drain(uint32_t bar, uint32_t parity, long long sent, long long armed,
                                        unsigned long long limit_ns) const {
    const uint32_t mb = base + bar;
    if (sent < armed) mbar_complete_tx(mb, (uint32_t)(armed - sent));
    if (mbar_wait(mb, parity, limit_ns) && sent > armed) {
      mbar_arrive_expect(mb, (uint32_t)(sent - armed));
      mbar_wait(mb, parity ^ 1u, limit_ns);
    }
  }
};

// acc += (or -=) sum of val * buf[col] over one slice: lane l gets the sums of
// the row l >> lg (every lane of the row the same).  Steps go by fours, the
// next four's loads in flight while four are gathered and added; the last
// w mod 4 are loaded first and added last, in a loop of their own: a float64
// operation whose predicate is off still takes its slot of the float64 pipe
// (16 clocks of an SM), so no operation here is predicated.  Slices of
// kResWide steps and more use two accumulators: the chain of dependent float64
// operations (68 clocks each) is what a lone warp waits for, and the extra
// addition is a small part of so long a row.
constexpr int kResWide = 12;
template <bool kNegate, typename TV>
__device__ __forceinline__ TV res_fma(TV a, TV x, TV acc) {
  return kNegate ? fmadd(-a, x, acc) : fmadd(a, x, acc);
}
template <int NB, bool kNegate, typename TV, typename TX>
__device__ __forceinline__ void res_dot(const ResSlice& s, const TV* __restrict__ val,
                                        const uint16_t* __restrict__ col, const TX* const (&buf)[NB],
                                        TV (&acc)[NB]) {
  const int lane = threadIdx.x & 31, w = res_steps(s.wgr), lg = res_lg(s.wgr);
  const TV* v = val + s.off + lane;
  const uint16_t* c = col + s.off + lane;
  const int full = w & ~3;
  TV a[4], ta[3];
  int j[4], tj[3];
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    a[e] = TV(0);
    j[e] = 0;
    if (full) {
      a[e] = __ldg(v + e * 32);
      j[e] = __ldg(c + e * 32);
    }
  }
#pragma unroll
  for (int e = 0; e < 3; ++e) {
    ta[e] = TV(0);
    tj[e] = 0;
    if (full + e < w) {
      ta[e] = __ldg(v + (full + e) * 32);
      tj[e] = __ldg(c + (full + e) * 32);
    }
  }
  // four steps: the values and columns in a, j; f adds value * entry to step e's sum
  auto four = [&](int k, auto&& f) {
    TV g[NB][4], ca[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      ca[e] = a[e];
#pragma unroll
      for (int b = 0; b < NB; ++b) g[b][e] = (TV)buf[b][j[e]];
    }
    if (k + 4 < full) {
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        a[e] = __ldg(v + (k + 4 + e) * 32);
        j[e] = __ldg(c + (k + 4 + e) * 32);
      }
    }
#pragma unroll
    for (int e = 0; e < 4; ++e)
#pragma unroll
      for (int b = 0; b < NB; ++b) f(e, b, ca[e], g[b][e]);
  };
  if (w >= kResWide) {
    TV acc2[NB];
#pragma unroll
    for (int b = 0; b < NB; ++b) acc2[b] = TV(0);
#pragma unroll 1
    for (int k = 0; k < full; k += 4)
      four(k, [&](int e, int b, TV x, TV y) {
        if (e & 1) acc2[b] = res_fma<kNegate>(x, y, acc2[b]);
        else acc[b] = res_fma<kNegate>(x, y, acc[b]);
      });
#pragma unroll
    for (int b = 0; b < NB; ++b) acc[b] += acc2[b];
  } else {
#pragma unroll 1
    for (int k = 0; k < full; k += 4)
      four(k, [&](int, int b, TV x, TV y) { acc[b] = res_fma<kNegate>(x, y, acc[b]); });
  }
#pragma unroll 1
  for (int e = full; e < w; ++e) {
#pragma unroll
    for (int b = 0; b < NB; ++b) acc[b] = res_fma<kNegate>(ta[0], (TV)buf[b][tj[0]], acc[b]);
    ta[0] = ta[1], tj[0] = tj[1];
    ta[1] = ta[2], tj[1] = tj[2];
  }
  if (lg) {  // warp-uniform
#pragma unroll 1
    for (int o = 1 << (lg - 1); o > 0; o >>= 1)
#pragma unroll
      for (int b = 0; b < NB; ++b) acc[b] += __shfl_xor_sync(0xffffffffu, acc[b], o);
  }
}

// One matrix of an LP as a CTA sees it; f(slice, row of this lane or -1) for
// the CTA's slices of this warp (row -1: a lane without a row of its own).
// The first slice's descriptor stays in registers, the next one's is loaded
// ahead.  empty(): the warp has no slice.
struct ResMat {
  const ResSlice* sl;
  const uint16_t* col;
  int slices, s0;
  int4 first;
  __device__ __forceinline__ ResMat(const ResSlice* sl_, const uint16_t* col_, int n, int rank, int C)
      : sl(sl_), col(col_), slices(n), s0(rank + (int)(threadIdx.x >> 5) * C) {
    first = s0 < n ? __ldg(reinterpret_cast<const int4*>(sl + s0)) : make_int4(0, 0, 0, 0);
  }
  __device__ __forceinline__ bool empty() const { return s0 >= slices; }
  template <int C, class F>
  __device__ __forceinline__ void each(F&& f) const {
    const int lane = threadIdx.x & 31;
    int4 q = first;
    for (int s = s0; s < slices; s += kResWarps * C) {
      const ResSlice d{q.x, q.y, q.z, q.w};
      if (s + kResWarps * C < slices) q = __ldg(reinterpret_cast<const int4*>(sl + s + kResWarps * C));
      const int lg = res_lg(d.wgr), row = lane >> lg;
      f(d, (lane & ((1 << lg) - 1)) == 0 && row < res_rows(d.wgr) ? row : -1);
    }
  }
};

// a warp that no vector has to arrive for (see the head of this file)
__device__ __forceinline__ bool res_idle(const ResMat& a, const ResMat& b) {
  return threadIdx.x >= 32 && a.empty() && b.empty();
}

// Sums of NQ quantities over the cluster, the same bits on every CTA: the
// block's sums to every CTA's record of this rank, a cluster barrier, then the
// records in rank order into out[0..NQ) (shared).  `flag` (thread 0's) of rank
// 0 is returned to every thread.  Ends with a block barrier; the caller meets
// a cluster barrier before the next call.
template <int NQ, int C>
__device__ __forceinline__ bool res_reduce(const ResCluster<C>& cl, const ResSmem& L,
                                           unsigned char* smem, double (&v)[NQ], double* out,
                                           bool flag = false) {
  double* rec = reinterpret_cast<double*>(smem + L.rec);
  double* red = reinterpret_cast<double*>(smem + L.red);
  block_sum_scatter<kResThreads, NQ>(v, red, out);
  if (threadIdx.x < NQ) cl.push(L.rec + (uint32_t)(cl.rank * 18 + threadIdx.x) * 8u, out[threadIdx.x]);
  if (threadIdx.x == 0) cl.push(L.rec + (uint32_t)(cl.rank * 18 + 16) * 8u, flag ? 1.0 : 0.0);
  cl.sync();
  if (threadIdx.x < NQ) {
    double t = rec[threadIdx.x];
#pragma unroll
    for (int r = 1; r < C; ++r) t += rec[r * 18 + threadIdx.x];
    out[threadIdx.x] = t;
  }
  const bool f = rec[16] != 0.0;
  __syncthreads();
  return f;
}

// Exchanges of an iteration that needs sums besides the two vectors (the power
// iteration, the conjugate gradients): barrier 0 counts X, 1 Y, 2 and 3 the
// records of two sums.  Each barrier goes through one phase per iteration.  A
// CTA may be one exchange ahead of another, never two: each sum waits for every
// CTA's part, so a record is read everywhere before its slot is written again.
// All warps wait for the sums (each ends with a block barrier, and its next
// phase needs records sent behind it); idle ones do not wait for X and Y.
template <int C>
struct ResExchange {
  static constexpr int kFlags = 4 * kResMaxC, kCounts = 5 * kResMaxC;  // in the records, behind the sums
  const ResCluster<C>& cl;
  const ResSmem& L;
  unsigned char* smem;
  unsigned long long wait_ns;
  uint32_t bytes_x, bytes_y;
  int nq0, nq1;        // quantities of the two sums
  uint32_t extra;      // bytes every phase expects and nobody sends (wait_test)
  bool idle;           // this warp (res_idle)
  uint32_t phase = 0;
  bool lost = false;  // a wait ran out (uniform in a warp, which sends nothing more)
  uint32_t sent[4] = {}, seen[4] = {};  // per barrier: values sent, phases seen complete
  __device__ __forceinline__ ResExchange(const ResCluster<C>& c, const ResSmem& l, unsigned char* s,
                                         unsigned long long limit, uint32_t bx, uint32_t by,
                                         int q0, int q1, uint32_t extra_, bool idle_)
      : cl(c), L(l), smem(s), wait_ns(limit), bytes_x(bx), bytes_y(by), nq0(q0), nq1(q1), extra(extra_),
        idle(idle_) {
    if (C > 1 && threadIdx.x < kResMaxC) reinterpret_cast<double*>(smem + L.rec)[kFlags + threadIdx.x] = 0.0;
    if (C > 1 && threadIdx.x == 0)
      for (int b = 0; b < 4; ++b) {
        mbar_init(cl.base + L.bar + 8u * b);
        mbar_arrive_expect(cl.base + L.bar + 8u * b, expect(b));
      }
  }
  __device__ __forceinline__ uint32_t expect(int b) const {
    return extra + (b == 0 ? bytes_x : b == 1 ? bytes_y : (uint32_t)(C * 8 * (b == 2 ? nq0 : nq1)));
  }
  __device__ __forceinline__ void send_x(int p, double v) {
    if (lost) return;
    cl.send(L.X + 8u * p, L.bar, v);
    sent[0] += 1;
  }
  __device__ __forceinline__ void send_y(int p, double v) {
    if (lost) return;
    cl.send(L.Y + 8u * p, L.bar + 8u, v);
    sent[1] += 1;
  }
  // this rank's record of quantity q, by a whole warp: lane r's to rank r
  __device__ __forceinline__ void send_record(int slot, int q, double v) {
    if (lost) return;
    if ((threadIdx.x & 31) < C)
      cl.send_to(threadIdx.x & 31, L.rec + (uint32_t)(slot * 2 * kResMaxC + q * kResMaxC + cl.rank) * 8u,
                 L.bar + 16u + 8u * slot, v);
    sent[2] += slot == 0;
    sent[3] += slot != 0;
  }
  __device__ __forceinline__ void wait(int b, uint32_t parity) {
    if (lost || (idle && b < 2)) return;
    lost = !cl.arrived(L.bar + 8u * b, parity, expect(b), wait_ns);
#pragma unroll
    for (int e = 0; e < 4; ++e) seen[e] += !lost && e == b;
  }
  __device__ __forceinline__ void wait(int b) {
    if constexpr (C == 1)
      __syncthreads();
    else
      wait(b, phase);
  }
  // NQ sums over the cluster, the same bits in every thread; slot 0 or 1, each
  // once per iteration.  The threads' shares go through shared memory to one
  // warp per quantity (16 values a lane, then a tree): every warp summing its
  // own by shuffles took 5 float64 operations of 16 clocks per warp and
  // quantity, 3600 clocks a sum; this takes about 1100.  What follows from a
  // total (a quotient, a root, a test) is taken there too, once instead of by
  // all 16 warps: fin(quantity, total, o) sets o[0..2], which every thread gets
  // in res[quantity][0..2].
  template <int NQ, class F>
  __device__ __forceinline__ void sum(const double (&v)[NQ], int slot, double (&res)[NQ][3], F&& fin) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    double* red = reinterpret_cast<double*>(smem + L.red);
    double* out = red + 2 * kResThreads;  // the totals
    const double* rec = reinterpret_cast<const double*>(smem + L.rec) + slot * 2 * kResMaxC;
#pragma unroll
    for (int q = 0; q < NQ; ++q) red[q * kResThreads + threadIdx.x] = v[q];
    __syncthreads();
    if (warp < NQ) {
      double t = block_share(red + warp * kResThreads + lane);
      send_record(slot, warp, t);
      if (C > 1) {
        // the records of every CTA, in a tree
        wait(2 + slot);
        double r = lane < C ? rec[warp * kResMaxC + lane] : 0.0;
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) r += __shfl_xor_sync(0xffffffffu, r, o);
        t = r;
      }
      if (lane == 0) {
        double o[3];
        fin(warp, t, o);
        out[4 * warp] = o[0];
        out[4 * warp + 1] = o[1];
        out[4 * warp + 2] = o[2];
      }
    } else if (C > 1) {
      wait(2 + slot);
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
      res[q][0] = out[4 * q];
      res[q][1] = out[4 * q + 1];
      res[q][2] = out[4 * q + 2];
    }
  }
  // The same in two parts: the last NQ warps add the CTA's shares and send them
  // in sum_begin; in sum_end, later in the loop, they add the CTAs' and call fin
  // (o[0..1]).  `slot` alternates between iterations, so a record is read before
  // its slot is written again although a CTA may be an iteration ahead; `parity`
  // is that of the slot's uses.  sum_end: whether a warp's wait ran out.
  template <int NQ>
  __device__ __forceinline__ void sum_begin(const double (&v)[NQ], int slot) {
    const int lane = threadIdx.x & 31, q = (int)(threadIdx.x >> 5) - (kResWarps - NQ);
    double* red = reinterpret_cast<double*>(smem + L.red);
#pragma unroll
    for (int e = 0; e < NQ; ++e) red[e * kResThreads + threadIdx.x] = v[e];
    __syncthreads();
    if (q < 0) return;
    send_record(slot, q, block_share(red + q * kResThreads + lane));
  }
  template <int NQ, class F>
  __device__ __forceinline__ bool sum_end(int slot, uint32_t parity, double (&res)[NQ][2], F&& fin) {
    const int lane = threadIdx.x & 31, q = (int)(threadIdx.x >> 5) - (kResWarps - NQ);
    double* out = reinterpret_cast<double*>(smem + L.red) + 2 * kResThreads;
    const double* rec = reinterpret_cast<const double*>(smem + L.rec) + slot * 2 * kResMaxC;
    if (C > 1) wait(2 + slot, parity);
    if (q >= 0) {
      double r = lane < C ? rec[q * kResMaxC + lane] : 0.0;
#pragma unroll
      for (int o = C / 2; o > 0; o >>= 1) r += __shfl_xor_sync(0xffffffffu, r, o);
      if (lane == 0) {
        double o[2];
        fin(q, r, o);
        out[4 * q] = o[0];
        out[4 * q + 1] = o[1];
      }
    }
    const bool ran_out = __syncthreads_or(lost);
#pragma unroll
    for (int e = 0; e < NQ; ++e) {
      res[e][0] = out[4 * e];
      res[e][1] = out[4 * e + 1];
    }
    return ran_out;
  }
  // the sum of 512 shares, 32 apart, of this lane and of its warp
  __device__ __forceinline__ double block_share(const double* mine) const {
    double t[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      t[e] = mine[e * 32];
#pragma unroll
      for (int k = 1; k < kResWarps / 4; ++k) t[e] += mine[(e + 4 * k) * 32];
    }
    t[0] = (t[0] + t[1]) + (t[2] + t[3]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) t[0] += __shfl_xor_sync(0xffffffffu, t[0], o);
    return t[0];
  }
  // whether the loop ends, the same for all of the CTA's threads (after a lost
  // wait its warps may have read different sums)
  __device__ __forceinline__ bool ends(bool stop) const { return __syncthreads_or(stop || lost); }
  // ends an iteration that used every barrier once
  __device__ __forceinline__ void next() { phase ^= 1u; }
  // Ends the kernel's exchanges (all threads of all CTAs): whether a wait ran out
  // in any CTA of the cluster.  Without one, everything sent has arrived, since
  // every CTA has waited for it.  With one, the CTAs tell each other how much
  // they have sent, and each waits for what is still on its way to it.
  __device__ __forceinline__ bool finish() {
    if constexpr (C == 1) return false;
    const double* rec = reinterpret_cast<const double*>(smem + L.rec);
    if (__syncthreads_or(lost) && threadIdx.x == 0) cl.push(L.rec + (uint32_t)(kFlags + cl.rank) * 8u, 1.0);
    cl.sync();
    bool any = false;
#pragma unroll
    for (int q = 0; q < C; ++q) any |= rec[kFlags + q] != 0.0;
    if (!any) return false;
    double v[4];
#pragma unroll
    for (int b = 0; b < 4; ++b)  // (a record is sent to each CTA by a lane of its own)
      v[b] = b < 2 || (threadIdx.x & 31) == 0 ? (double)sent[b] : 0.0;
    double* red = reinterpret_cast<double*>(smem + L.red);
    double* mine = red + 2 * kResThreads;
    block_sum_scatter<kResThreads, 4>(v, red, mine);
    if (threadIdx.x < 4) cl.push(L.rec + (uint32_t)(kCounts + 4 * cl.rank + threadIdx.x) * 8u, mine[threadIdx.x]);
    cl.sync();
    if (threadIdx.x == 0)
#pragma unroll
      for (int b = 0; b < 4; ++b) {
        double all = 0.0;
        for (int q = 0; q < C; ++q) all += rec[kCounts + 4 * q + b];
        cl.drain(L.bar + 8u * b, seen[b] & 1u, 8ll * (long long)all, (1ll + seen[b]) * expect(b), wait_ns);
      }
    return true;
  }
};

#define RES_DISPATCH_C(c, ...)  \
  switch (c) {                  \
    case 1: {                   \
      constexpr int C_ = 1;     \
      __VA_ARGS__;              \
    } break;                    \
    case 2: {                   \
      constexpr int C_ = 2;     \
      __VA_ARGS__;              \
    } break;                    \
    case 4: {                   \
      constexpr int C_ = 4;     \
      __VA_ARGS__;              \
    } break;                    \
    case 8: {                   \
      constexpr int C_ = 8;     \
      __VA_ARGS__;              \
    } break;                    \
    default: {                  \
      constexpr int C_ = 16;    \
      __VA_ARGS__;              \
    } break;                    \
  }

inline cudaLaunchConfig_t res_config(int C, int lps, size_t smem, cudaStream_t s,
                                     cudaLaunchAttribute* attr) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(lps * C);
  cfg.blockDim = dim3(kResThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  attr->id = cudaLaunchAttributeClusterDimension;
  attr->val.clusterDim.x = C;
  attr->val.clusterDim.y = attr->val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cfg;
}

// ---------------------------------------------------------------------------
// building and launching (resident.cu)
// ---------------------------------------------------------------------------
struct ResBuild {
  ResLp* lp;
  const int32_t *a_rp, *t_rp;   // stacked row pointers
  ResSlice *a_sl, *t_sl;        // slices of LP l at m_off / n_off (at most one per row)
  uint16_t *ord_m, *ord_n;      // local row / column at a position
  uint16_t *pos_m, *pos_n;      // position of a local row / column
  long long* elems;             // [2 lp]: elements of A~, A~^T
  int32_t* longest;             // the longest row of any matrix
};

// values and columns of the slices: a warp per slice, the matrices in y;
// entries past a row's end: value 0 and the column of the slot that holds 0
struct ResFill {
  const ResLp* lp;
  const int32_t *a_rp, *t_rp, *a_col, *t_col;  // columns in the stacked numbering
  const double *a_val, *t_val;
  const int32_t *a_src, *t_src;  // NULL, or where the values of entry k are
  const ResSlice *a_sl, *t_sl;
  const uint16_t *ord_m, *ord_n, *pos_m, *pos_n;
  uint16_t *a_c, *t_c;   // NULL: columns are in place
  double *a_v, *t_v;
  float *a_f, *t_f;      // NULL: no float32 copy
};
void launch_res_sort(const ResBuild& B, int count, cudaStream_t s);
void launch_res_fill(const ResFill& F, int count, int max_slices, cudaStream_t s);

// ---------------------------------------------------------------------------
// the solve (resident_solve.cuh)
// ---------------------------------------------------------------------------
template <typename T>
struct ResSolve {
  const ResLp* lp;
  const int32_t* list;  // LPs of this launch, one per cluster
  const ResSlice *a_sl, *t_sl;
  const uint16_t *a_col, *t_col, *ord_m, *ord_n;
  const T *a_val, *t_val;
  const double *a_val64, *t_val64;
  IterBuffers<T> B;       // the state in natural order
  int32_t* active;        // LPs not finished
  unsigned long long slice_ns;
  unsigned long long wait_ns;  // bound of a wait for another CTA's vector
  uint32_t tx_extra;           // bytes each such wait expects and nobody sends (wait_test)
  int32_t* err;                // 1 once such a wait ran out
};

template <typename T>
const void* res_solve_kernel(int C, bool halpern);
template <typename T>
cudaError_t launch_res_solve(const ResSolve<T>& A, int C, int lps, size_t smem, bool halpern,
                             cudaStream_t s);

}  // namespace pdhg
