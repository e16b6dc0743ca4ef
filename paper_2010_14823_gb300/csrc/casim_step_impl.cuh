// Definitions behind casim_step.cuh, for the translation units that
// instantiate a configuration's kernels.
#pragma once

#include <type_traits>

#include "casim_step.cuh"

namespace casim_dev {

// Threads that share a column, each a segment of its levels (a power of two;
// 1: one thread per column).  A segment costs one extra level (its upper
// neighbour, for the flux into it), so the column is split only as far as the
// warps still fit in one resident wave, and into no more segments than it has
// pairs of levels.  Measured, mixed cold step at 60 levels, 1 / 2 / 4 / 8 /
// 16 / 32 segments: 20 000 columns 172 / 120 / 90 / 93 / 101 / 124 us, 5 000
// columns - / 92 / 58 / 42 / 36 / 40 us; 256 columns x 50 levels 114 / 69 /
// 40 / 28 / 22 / 16 us.  Beyond a wave splitting loses: 65 536 columns x 100
// triple-moment 837 / 985 / 937 us, 262 144 x 150 cold 1927 / 2022 / 2060 us.
// A state in host memory saturates the host link with fewer warps
// (20 000 x 60: 834 / 840 / 853 us).
inline int step_segments(int ncols, int nlev, int nsm, int blocks_per_sm, bool line) {
  const long long warps = (ncols + 31) / 32, room = line ? 1024 : (long long)nsm * blocks_per_sm * (kBlock / 32);
  int n = 1;
  while (n < 32 && 2 * n <= nlev && 2 * n * warps <= room) n *= 2;
  return n;
}

// grid.x column groups; the levels of a column shared by clusters of grid.y blocks
template <class K>
cudaError_t step_launch(K kernel, dim3 grid, size_t smem, cudaStream_t st, const KArgs &a, const KParams &kp,
                        double *tend) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(kBlock);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = 1;
  at[0].val.clusterDim.y = grid.y;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = grid.y > 1 ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kernel, a, kp, tend);
}

template <class M>
cudaError_t step_allow_smem() {
  cudaError_t e = cudaSuccess;
  auto allow = [&](auto *kernel, size_t bytes) {
    if (e == cudaSuccess) e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  };
  allow(k_step<M, false>, step_smem_bytes<M, false, false>(kMaxLev));
  allow(k_step<M, true>, step_smem_bytes<M, true, false>(kMaxLev));
  allow(k_step<M, false, false, true>, step_smem_bytes<M, false, false>(kMaxLev));
  allow(k_step<M, false, false, false, true>, step_smem_bytes<M, false, true>(kMaxLev));
  allow(k_step<M, true, false, false, true>, step_smem_bytes<M, true, true>(kMaxLev));
  allow(k_step<M, false, false, true, true>, step_smem_bytes<M, false, true>(kMaxLev));
  return e;
}

template <class PMix, class PF64>
cudaError_t StepKernels<PMix, PF64>::allow_smem() {
  cudaError_t e = step_allow_smem<PMix>();
  if constexpr (std::is_same<PMix, PolicyMix>::value)
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(k_step<PMix, false, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               (int)step_smem_bytes<PMix, false, false>(kMaxLev));
  return e;
}

template <class PMix, class PF64>
cudaError_t StepKernels<PMix, PF64>::launch(const StepLaunch &l, const KArgs &args, const KParams &kp) {
  KArgs a = args;
  const bool line = l.line && l.mixed;
  const dim3 whole((unsigned)((a.ncols + kBlock - 1) / kBlock));
  if constexpr (std::is_same<PMix, PolicyMix>::value) {
    // the statistics build (a CASIM_STATS context: standard configuration)
    if (a.stats && !l.tend)
      return l.mixed ? step_launch(k_step<PMix, false, true>, whole, step_smem_bytes<PMix, false, false>(a.nlev),
                                   l.stream, a, kp, nullptr)
                     : step_launch(k_step<PF64, false, true>, whole, step_smem_bytes<PF64, false, false>(a.nlev),
                                   l.stream, a, kp, nullptr);
  }
  const int n = step_segments(a.ncols, a.nlev, l.nsm, l.mixed ? PMix::kMinBlocks : PF64::kMinBlocks, line);
  auto go = [&](auto *one, auto *split, size_t smem1, size_t smem) {
    if (n == 1) return step_launch(one, whole, smem1, l.stream, a, kp, l.tend);
    a.segs = n < kBlock / 32 ? n : kBlock / 32;   // a warp per segment in the block, the rest over a cluster
    const int cols = kBlock / a.segs;
    return step_launch(split, dim3((unsigned)((a.ncols + cols - 1) / cols), (unsigned)(n / a.segs)), smem, l.stream, a,
                       kp, l.tend);
  };
#define CASIM_STEP_PAIR(M, tend, line)                                                                \
  go(k_step<M, tend, false, line>, k_step<M, tend, false, line, true>, step_smem_bytes<M, tend, false>(a.nlev), \
     step_smem_bytes<M, tend, true>(a.nlev))
  if (l.mixed) {
    if (l.tend) return CASIM_STEP_PAIR(PMix, true, false);
    if (line) return CASIM_STEP_PAIR(PMix, false, true);
    return CASIM_STEP_PAIR(PMix, false, false);
  }
  if (l.tend) return CASIM_STEP_PAIR(PF64, true, false);
  return CASIM_STEP_PAIR(PF64, false, false);
#undef CASIM_STEP_PAIR
}

}  // namespace casim_dev
