// Host side shared by the on-chip solve and the on-chip conjugate gradients:
// launch groups (LPs of one cluster size), their streams, and the choice of
// cluster sizes.
#pragma once
#include <functional>
#include <vector>

#include "context.h"
#include "resident.cuh"

namespace pdhg {

struct ResGroup {
  int C, first, count;  // LPs list[first..first + count)
  size_t smem_solve = 0, smem_power = 0;
};

// the groups of a launch run side by side on streams of their own
struct ResStreams {
  cudaStream_t s[4] = {};
  cudaEvent_t fork = nullptr, join[4] = {};
  int have = 0;
  cudaError_t make(int groups) {
    cudaError_t e = cudaSuccess;
    if (groups > 1 && !fork) e = cudaEventCreateWithFlags(&fork, cudaEventDisableTiming);
    for (; have < groups - 1 && e == cudaSuccess; ++have) {
      e = cudaStreamCreateWithFlags(&s[have], cudaStreamNonBlocking);
      if (e == cudaSuccess) e = cudaEventCreateWithFlags(&join[have], cudaEventDisableTiming);
    }
    return e;
  }
  void free() {
    for (cudaStream_t q : s)
      if (q) cudaStreamDestroy(q);
    for (cudaEvent_t q : join)
      if (q) cudaEventDestroy(q);
    if (fork) cudaEventDestroy(fork);
    *this = ResStreams{};
  }
};

// launch(group, stream) for every group, between what the context's stream
// holds before and after
template <class F>
pdhg_status res_groups(pdhg_ctx* ctx, const std::vector<ResGroup>& groups, const ResStreams& side,
                       F&& launch) {
  if (groups.size() > 1) CK(cudaEventRecord(side.fork, ctx->stream));
  for (size_t g = 0; g < groups.size(); ++g) {
    cudaStream_t s = g == 0 ? ctx->stream : side.s[g - 1];
    if (g) CK(cudaStreamWaitEvent(s, side.fork, 0));
    CK(launch(groups[g], s));
    ctx->launches += 1;
    if (g) CK(cudaEventRecord(side.join[g - 1], s));
  }
  for (size_t g = 1; g < groups.size(); ++g) CK(cudaStreamWaitEvent(ctx->stream, side.join[g - 1], 0));
  return PDHG_OK;
}

// bytes beyond those sent that a wait between CTAs expects
inline uint32_t res_tx_extra(const pdhg_ctx* ctx) { return ctx->opt.wait_test ? 8u : 0u; }

std::vector<int> res_clusters(const pdhg_ctx* ctx, const std::vector<double>& ops, double min_ops,
                              const std::function<bool(int, int)>& fits);
std::vector<int32_t> res_order(const std::vector<ResLp>& lps, const std::vector<double>& ops);
bool res_fits(const void* f, int C, size_t smem, size_t smem_optin);

}  // namespace pdhg
