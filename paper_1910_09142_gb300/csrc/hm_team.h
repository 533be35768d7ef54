// Host side of a team: the thread-block cluster that works on one chain
// when a batch has fewer chains than the GPU has SMs.
//
// A chain's ops are serial, but the charge blocks of one split are not: a team
// shares out theta's tiles, the blocks (each decomposed by one CTA, the
// costliest first) and the absorb, and meets at three cluster barriers an op.
// Everything a CTA needs from another goes through the chain's own buffers in
// global memory.  A Markov step, one CTA -> a team: 4 chains of Lx = 4, 2W =
// 4, binary64, 206 -> 113 ms (8 CTAs); 8 mixed chains of Lx = 4, 30.4 -> 22.4
// ms (8); one METTS chain of small blocks, 22.1 -> 20.4 ms (8).
#pragma once

#include <cuda_runtime.h>

#include <mutex>

#include "hm_internal.h"

namespace hm {

// Bond caps up to here get one CTA a chain in every batch: a split has a few blocks
// of a few columns, and three cluster barriers cost more than they share out.
// us an op, one CTA and a team of 8 (1 to 70 chains): HM_FP64 cap 3 25 and 30, cap 9
// 37 and 41, cap 27 51 and 51, cap 64 97 to 119 and 88 to 108; HM_MIXED 37 and 40, 39 and 41,
// 46 and 46, 67 to 74 and 60 to 69.
constexpr int kTeamChiCap = 27;

// Largest cluster size of 8, 4 or 2 of which n are resident at once (most[e]:
// clusters of 2^e that fit), else 1.
inline int pick_team(const int (&most)[4], int n, int chi_cap) {
  if (chi_cap <= kTeamChiCap) return 1;
  for (int e = 3; e >= 1; --e)
    if (most[e] >= n) return 1 << e;
  return 1;
}

#if !defined(HM_HOST_EMULATION)
// Cluster size for n chains with bond caps up to chi_cap.  The occupancy answers
// are kept per device and kernel (at most four kernels).
inline int team_size(const void* kernel, int threads, size_t smem, int n, int chi_cap) {
  struct Known {
    const void* kernel;
    int dev, most[4];                       // clusters of 2, 4 and 8 that fit
  };
  static std::mutex mu;
  static Known known[16] = {};
  static int n_known = 0;
  if (2 * n > device_sm_count() || chi_cap <= kTeamChiCap) return 1;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return 1;
  std::lock_guard<std::mutex> lock(mu);
  Known* k = nullptr;
  for (int i = 0; i < n_known; ++i)
    if (known[i].kernel == kernel && known[i].dev == dev) k = &known[i];
  Known own = {kernel, dev, {0, 0, 0, 0}};
  if (!k) {
    for (int e = 1; e <= 3; ++e) {
      cudaLaunchAttribute at = {};
      at.id = cudaLaunchAttributeClusterDimension;
      at.val.clusterDim.x = 1u << e;
      at.val.clusterDim.y = at.val.clusterDim.z = 1;
      cudaLaunchConfig_t cfg = {};
      cfg.gridDim = dim3(1u << e);
      cfg.blockDim = dim3(threads);
      cfg.dynamicSmemBytes = smem;
      cfg.attrs = &at;
      cfg.numAttrs = 1;
      if (cudaOccupancyMaxActiveClusters(&own.most[e], kernel, &cfg) != cudaSuccess) {
        own.most[e] = 0;
        cudaGetLastError();                 // an unsupported size is not an error of the launch
      }
    }
    k = &own;
    if (n_known < 16) {
      known[n_known] = own;
      k = &known[n_known++];
    }
  }
  return pick_team(k->most, n, chi_cap);
}

template <typename... P, typename... A>
int launch_team(void (*kernel)(BatchArg, OutArg, P...), const BatchArg& b, const OutArg& o, int team, int threads,
                size_t smem, void* stream, A... more) {
  cudaLaunchAttribute at = {};
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = team;
  at.val.clusterDim.y = at.val.clusterDim.z = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)b.n * team);
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = (cudaStream_t)stream;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, b, o, P(more)...) == cudaSuccess ? HM_OK : HM_ERR_CUDA;
}
#endif

}  // namespace hm
