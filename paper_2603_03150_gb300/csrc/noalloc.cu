// Algorithm 1 (Section 3.1) centered start point on caller-provided device
// vectors with no device allocation (pdhg_centered_point_noalloc in
// include/pdhg.h).
//
// Some callers cannot call cudaMalloc: an interior-point solver that owns a
// fixed device memory pool and must not grow it, or a host thread that must
// not take the device allocator's locks.  For them the scratch this
// computation needs -- one partial sum of x^T z per block -- lives in a file-scope __device__ array that every GPU which loads this
// library holds until the process exits.
#include <mutex>

#include "common.cuh"
#include "pdhg.h"
#include "resident.cuh"

namespace pdhg {
void set_error(const char* fmt, ...);
}

namespace {

constexpr int kNaThreads = 256;
constexpr int kNaPerBlock = 2048;   // entries of x^T z reduced by one block
constexpr int kNaMaxBlocks = 4096;  // partial-sum slots
// Blocks of the second pass, two per SM of a GB300: an entry's quotients bound it
// (about 24 operations of the float64 pipe, which 16 warps per SM keep busy), and
// every block adds the partial sums again (300,000 / 1,000,000 / 8,388,608
// entries, in strides of the grid: 304 blocks 26.6 / 69.7 / 519 us, 608 26.7 / 71.7
// / 521, 1216 28.7 / 76.2 / 522).
constexpr int kNaApplyBlocks = 304;
constexpr long long kNaMaxN = (long long)kNaPerBlock * kNaMaxBlocks;  // 8,388,608

// Per-block partial sums of x^T z.  Every call writes each slot it reads before reading it, so nothing has to
// be cleared between calls.  32 KB per device.
static __device__ __align__(256) double g_na_scratch[kNaMaxBlocks];

// sum of x z over [base, end) by one block, in thread 0
__device__ __forceinline__ double na_block_sum(int base, int end, const double* __restrict__ x,
                                               const double* __restrict__ z, double* red) {
  double acc = 0.0;
  for (int i = base + threadIdx.x; i < end; i += kNaThreads) acc += x[i] * z[i];
  const double v[1] = {acc};
  double o[1];
  pdhg::block_sum<kNaThreads, 1>(v, o, red);
  return o[0];
}

// n <= kNaSmall: one launch, a cluster of 8 blocks whose sums of x^T z go
// through distributed shared memory.  Three launches took 14.5 us call after
// call at any of these sizes and one block of 256 threads 10.4 / 14.6 / 24.3 at
// 500 / 1000 / 2000 entries (an entry's quotients keep an SM's float64 pipe for
// 18 clocks); the cluster takes 8.3 up to 2048 entries and 10.4 up to 4096, the two
// launches above 10.3 at 4097.
constexpr int kNaCluster = 8, kNaSmall = 4096;
__global__ void __cluster_dims__(kNaCluster, 1, 1) __launch_bounds__(kNaThreads)
    k_na_small(int n, const double* __restrict__ x, const double* __restrict__ z, double mu_min,
               double delta, double alpha, double* mu_out, double* __restrict__ x_out,
               double* __restrict__ z_out) {
  constexpr int K = kNaSmall / (kNaCluster * kNaThreads);
  __shared__ double part[kNaCluster], red[kNaThreads / 32], mu_s;
  const pdhg::ResCluster<kNaCluster> cl(part);
  const int first = cl.rank * kNaThreads + threadIdx.x;
  double xs[K], zs[K];
#pragma unroll
  for (int k = 0; k < K; ++k) {
    const int j = first + k * kNaCluster * kNaThreads;
    xs[k] = j < n ? x[j] : 0.0;
    zs[k] = j < n ? z[j] : 0.0;
  }
  cl.sync();  // every block runs: its shared memory may be written
  double acc[1] = {0.0}, sum[1];
#pragma unroll
  for (int k = 0; k < K; ++k) acc[0] += xs[k] * zs[k];
  pdhg::block_sum<kNaThreads, 1>(acc, sum, red);
  if (threadIdx.x == 0) cl.push((uint32_t)cl.rank * 8u, sum[0]);
  cl.sync();
  if (threadIdx.x == 0) {
    const double s = ((part[0] + part[1]) + (part[2] + part[3])) + ((part[4] + part[5]) + (part[6] + part[7]));
    mu_s = fmax(s / (double)n, mu_min);
    if (mu_out && cl.rank == 0) *mu_out = mu_s;
  }
  __syncthreads();
#pragma unroll 1
  for (int k = 0; k < K; ++k) {
    const int j = first + k * kNaCluster * kNaThreads;
    if (j >= n) break;
    pdhg::centered_pair(mu_s, delta, alpha, xs[0], zs[0]);
    x_out[j] = xs[0];
    z_out[j] = zs[0];
    xs[0] = xs[K - 1], zs[0] = zs[K - 1];
  }
}
static_assert(kNaSmall == 2 * kNaCluster * kNaThreads, "an entry or two per thread");

// partial sums of x^T z
__global__ void __launch_bounds__(kNaThreads)
    k_na_partial(int n, const double* __restrict__ x, const double* __restrict__ z, double* scratch) {
  __shared__ double red[kNaThreads / 32];
  const int base = blockIdx.x * kNaPerBlock;
  const double s = na_block_sum(base, min(n, base + kNaPerBlock), x, z, red);
  if (threadIdx.x == 0) scratch[blockIdx.x] = s;
}

// mu, which the first warp of every block adds from the partial sums (one order
// in all of them), and Algorithm 1's per-entry update (Section 3.1).  Nothing of a
// call outlives it: a count of finished blocks, which would let the last one of
// k_na_partial add the sums, would be wrong for good after two calls that overlap
// (and took longer: 4097 / 50,000 / 300,000 entries 12.3 / 14.4 / 27.7 us against
// 10.3 / 12.3 / 26.6).
__global__ void __launch_bounds__(kNaThreads)
    k_na_apply(int n, const double* __restrict__ x, const double* __restrict__ z,
               const double* scratch, int nparts, double mu_min, double delta, double alpha,
               double* mu_out, double* __restrict__ x_out, double* __restrict__ z_out) {
  __shared__ double mu_s;
  if (threadIdx.x < 32) {
    double s[4] = {0.0, 0.0, 0.0, 0.0};
    for (int p = threadIdx.x; p < nparts; p += 128)
#pragma unroll
      for (int e = 0; e < 4; ++e)
        if (p + 32 * e < nparts) s[e] += __ldcg(scratch + p + 32 * e);
    double t = (s[0] + s[1]) + (s[2] + s[3]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    t = fmax(t / (double)n, mu_min);
    if (threadIdx.x == 0) {
      mu_s = t;
      if (mu_out && blockIdx.x == 0) *mu_out = t;
    }
  }
  __syncthreads();
  const double mu = mu_s;
  // a run of entries per block, in whole warps: SMs get the same share of them
  // (strides of the grid leave a last round to some of the blocks: 358,000
  // entries 32.8 us against 30.7)
  const int per = ((n + (int)gridDim.x - 1) / (int)gridDim.x + 31) & ~31;
  const int first = (int)blockIdx.x * per, end = min(n, first + per);
  for (int j = first + threadIdx.x; j < end; j += kNaThreads) {
    double xp = x[j], zp = z[j];
    pdhg::centered_pair(mu, delta, alpha, xp, zp);
    x_out[j] = xp;
    z_out[j] = zp;
  }
}

// Device address of g_na_scratch, looked up once per device (in the device's
// primary context; a cudaDeviceReset would leave it stale, and the header
// rules that out).
std::mutex g_na_mutex;
constexpr int kNaMaxDevices = 256;
double* g_na_ptr[kNaMaxDevices] = {};

}  // namespace

extern "C" pdhg_status pdhg_centered_point_noalloc(int32_t n, const double* x, const double* z,
                                                   double mu_min, double delta_max,
                                                   double alpha_min, double* x_out, double* z_out,
                                                   double* mu_target, void* stream) {
  if (n < 1 || (long long)n > kNaMaxN) {
    pdhg::set_error("pdhg_centered_point_noalloc: n = %d outside [1, %lld] (the static scratch "
                    "holds %d partial sums of %d entries each)",
                    n, kNaMaxN, kNaMaxBlocks, kNaPerBlock);
    return PDHG_INVALID_ARG;
  }
  if (!x || !z || !x_out || !z_out) {
    pdhg::set_error("pdhg_centered_point_noalloc: x, z, x_out and z_out must be device pointers");
    return PDHG_INVALID_ARG;
  }
  if (!(mu_min > 0.0) || !(delta_max >= 0.0) || !(alpha_min > 0.0)) {
    pdhg::set_error("pdhg_centered_point_noalloc: need mu_min > 0, delta_max >= 0, alpha_min > 0");
    return PDHG_INVALID_ARG;
  }
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess || dev < 0 || dev >= kNaMaxDevices) {
    pdhg::set_error("pdhg_centered_point_noalloc: cudaGetDevice failed: %s", cudaGetErrorString(e));
    return PDHG_CUDA_ERROR;
  }
  double* scratch = nullptr;
  {
    std::lock_guard<std::mutex> lock(g_na_mutex);
    if (!g_na_ptr[dev]) {
      // set-up on the first call on this device (the current device)
      void* p = nullptr;
      e = cudaGetSymbolAddress(&p, g_na_scratch);
      if (e != cudaSuccess || !p) {
        pdhg::set_error("pdhg_centered_point_noalloc: cudaGetSymbolAddress failed: %s",
                        cudaGetErrorString(e));
        return PDHG_CUDA_ERROR;
      }
      g_na_ptr[dev] = static_cast<double*>(p);
    }
    scratch = g_na_ptr[dev];
  }
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const int nblocks = (int)((n + kNaPerBlock - 1) / kNaPerBlock);
  if (n <= kNaSmall) {
    k_na_small<<<kNaCluster, kNaThreads, 0, s>>>(n, x, z, mu_min, delta_max, alpha_min, mu_target, x_out,
                                                 z_out);
  } else {
    k_na_partial<<<nblocks, kNaThreads, 0, s>>>(n, x, z, scratch);
    int grid = (n + kNaThreads - 1) / kNaThreads;
    if (grid > kNaApplyBlocks) grid = kNaApplyBlocks;
    k_na_apply<<<grid, kNaThreads, 0, s>>>(n, x, z, scratch, nblocks, mu_min, delta_max, alpha_min, mu_target,
                                           x_out, z_out);
  }
  e = cudaGetLastError();
  if (e != cudaSuccess) {
    pdhg::set_error("pdhg_centered_point_noalloc: launch failed: %s", cudaGetErrorString(e));
    return PDHG_CUDA_ERROR;
  }
  return PDHG_OK;
}
