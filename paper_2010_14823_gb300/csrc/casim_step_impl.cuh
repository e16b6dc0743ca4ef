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
// levels (256 columns of 32 levels, 16 / 32 segments: 23.4 / 20.7 us; of 16
// levels, 8 / 16 segments: 23.7 / 20.4).  The wave is that of columns of a few
// hundred levels: at 1024 levels three blocks fit, not kMinBlocks, but fewer
// segments would be slower there (3 000 columns, 8 / 16 / 32 segments: 454 / 277 /
// 273 us; 12 000: 944 / 868 / 870).  Measured, mixed cold step at 60 levels, 1 / 2 / 4 / 8 /
// 16 / 32 segments: 20 000 columns 172 / 120 / 90 / 93 / 101 / 124 us, 5 000
// columns - / 92 / 58 / 42 / 36 / 40 us; 256 columns x 50 levels 114 / 69 /
// 40 / 28 / 22 / 16 us.  Beyond a wave splitting loses: 65 536 columns x 100
// triple-moment 837 / 985 / 937 us, 262 144 x 150 cold 1927 / 2022 / 2060 us.
// The warm forms with a third field stop at five blocks per SM, not at the wave's
// seven and eight: in steps of several substeps their full SMs leave the flux
// arrays too little cache (65 536 x 60, 1 / 2 segments, aerosol mass: dt = 1 s
// 199 / 187 us, dt = 10 s 385 / 660; sixth moments, 100 levels, dt = 10 s: 937 /
// 1223).
// A state in host memory saturates the host link with fewer warps
// (20 000 x 60: 834 / 840 / 853 us).
inline int step_segments(int ncols, int nlev, int nsm, int blocks_per_sm, bool line) {
  const long long warps = (ncols + 31) / 32, room = line ? 1024 : (long long)nsm * blocks_per_sm * (kBlock / 32);
  int n = 1;
  while (n < 32 && 2 * n <= nlev && 2 * n * warps <= room) n *= 2;
  return n;
}

// Blocks of half the threads, for a domain of one thread per column that fills
// no more than one resident wave: its blocks spread unevenly over the SMs
// (65 536 columns are 3.4 blocks of 128 per SM, so some SMs hold 16 warps and
// others 12), and the fullest SM sets the time.
// Measured (65 536 columns): source terms, 150 levels 985 -> 911 us; dt = 10 s,
// 100 levels 951 -> 929 us; 60 000 x 100 cold 415 -> 412 us; triple-moment
// 436 us either way at dt = 1 s and 60 levels, 1776 -> 1708 us at dt = 10 s and 100.
inline bool half_blocks(int warps, int nsm, int blocks_per_sm) {
  const int whole = (warps + 3) / 4, half = (warps + 1) / 2;
  if (whole > nsm * blocks_per_sm) return false;
  return 2 * ((half + nsm - 1) / nsm) < 4 * ((whole + nsm - 1) / nsm);   // warps of the fullest SM
}

// The FP64 sweep's segments per column group (1, 2, 4 or 8 blocks of a
// cluster, at least 4 levels each).  Four or eight, if that gives at most
// split_blocks blocks per SM (cold step: 1.5 resident waves); two, if they are
// resident at once, since twice two half columns take longer than one wave of
// whole ones.  Measured, cold step, us with 1 / 2 / 4 / 8 segments:
//   columns x levels   deep convection x 60        stratus x 150
//   1 824              577 / 404 / 378 / 327       938 /  589 /  575 /  475
//   2 400              537 / 370 / 382 / 394      1044 /  593 /  638 /  539
//   3 648              545 / 608 / 626 / 518      1044 /  902 /  964 /  732
//   4 864              546 / 609 / 696 / 662      1050 /  908 / 1132 /  908
//   6 400              856 /1065 / 855 / 814      1454 / 1693 / 1434 / 1164
//   9 600              888 /1171 /1168 /1153      1467 / 1758 / 1945 / 1635
inline int f64_segments(unsigned groups, int nlev, int nsm, int resident, int split_blocks) {
  for (int n = 8; n > 2; n /= 2)
    if (4 * n <= nlev && n * groups <= (unsigned)(nsm * split_blocks)) return n;
  return 8 <= nlev && 2 * groups <= (unsigned)(nsm * resident) ? 2 : 1;
}

// grid.x column groups; the levels of a column shared by clusters of grid.y blocks
template <class K>
cudaError_t step_launch(K kernel, dim3 grid, size_t smem, cudaStream_t st, const KArgs &a, const KParams &kp,
                        double *tend, int block = kBlock) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(block);
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

template <class PMix, class PF64>
cudaError_t StepKernels<PMix, PF64>::allow_smem() {
  cudaError_t e = cudaSuccess;
  auto allow = [&](auto *kernel, size_t bytes) {
    if (e == cudaSuccess) e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  };
  const size_t mixed = step_smem_bytes<PMix>(kMaxLev), fp64 = f64_smem_bytes<PF64>(kMaxLev);
  allow(k_step<PMix, false>, mixed);
  allow(k_step<PMix, true>, mixed);
  allow(k_step<PMix, false, false, true>, mixed);
  allow(k_step<PMix, false, false, false, true>, mixed);
  allow(k_step<PMix, true, false, false, true>, mixed);
  allow(k_step<PMix, false, false, true, true>, mixed);
  allow(k_step<PMix, false, false, false, false, kBlock / 2>, mixed);
  allow(k_step<PMix, true, false, false, false, kBlock / 2>, mixed);
  allow(k_step<PF64, false>, fp64);
  allow(k_step<PF64, true>, fp64);
  if constexpr (std::is_same<PMix, PolicyMix>::value) {
    allow(k_step<PMix, false, true>, mixed);
    allow(k_step<PF64, false, true>, f64_smem_bytes<PF64, true>(kMaxLev));
  }
  return e;
}

template <class PMix, class PF64>
cudaError_t StepKernels<PMix, PF64>::launch(const StepLaunch &l, const KArgs &args, const KParams &kp) {
  // the kernels' blocks per SM fit its shared memory (228 KB, 1 KB of each block reserved)
  static_assert(PF64::kMinBlocks * (f64_smem_bytes<PF64>(150) + 1024) <= 228 * 1024, "FP64 blocks per SM");
  static_assert(PMix::kMinBlocks * (step_smem_bytes<PMix>(150) + 1024) <= 228 * 1024, "mixed blocks per SM");
  KArgs a = args;
  const bool line = l.line && l.mixed;
  const unsigned groups = (unsigned)((a.ncols + kF64Cols - 1) / kF64Cols);   // FP64 blocks
  const dim3 whole((unsigned)((a.ncols + kBlock - 1) / kBlock));
  if constexpr (std::is_same<PMix, PolicyMix>::value) {
    // the statistics build (a CASIM_STATS context: standard configuration)
    if (a.stats && !l.tend)
      return l.mixed ? step_launch(k_step<PMix, false, true>, whole, step_smem_bytes<PMix>(a.nlev), l.stream, a, kp,
                                   nullptr)
                     : step_launch(k_step<PF64, false, true>, dim3(groups), f64_smem_bytes<PF64, true>(a.nlev), l.stream,
                                   a, kp, nullptr);
  }
  if (!l.mixed) {
    // FP64: blocks of 32 columns, a cluster of segments where they are few
    const dim3 grid(groups, (unsigned)f64_segments(groups, a.nlev, l.nsm, PF64::kMinBlocks, PF64::kSplitBlocks));
    const size_t smem = f64_smem_bytes<PF64>(a.nlev);
    return l.tend ? step_launch(k_step<PF64, true>, grid, smem, l.stream, a, kp, l.tend)
                  : step_launch(k_step<PF64, false>, grid, smem, l.stream, a, kp, nullptr);
  }
  const int n = step_segments(a.ncols, a.nlev, l.nsm, PMix::kSplitBlocks, line);
  const size_t smem = step_smem_bytes<PMix>(a.nlev);
  const bool half = n == 1 && !line && half_blocks((a.ncols + 31) / 32, l.nsm, PMix::kMinBlocks);
  auto go = [&](auto *one, auto *split, auto *small) {
    if (half)
      return step_launch(small, dim3((unsigned)((a.ncols + kBlock / 2 - 1) / (kBlock / 2))),
                         step_smem_bytes<PMix, kBlock / 2>(a.nlev), l.stream, a, kp, l.tend, kBlock / 2);
    if (n == 1) return step_launch(one, whole, smem, l.stream, a, kp, l.tend);
    a.segs = n < kBlock / 32 ? n : kBlock / 32;   // a warp per segment in the block, the rest over a cluster
    const int cols = kBlock / a.segs;
    return step_launch(split, dim3((unsigned)((a.ncols + cols - 1) / cols), (unsigned)(n / a.segs)), smem, l.stream, a,
                       kp, l.tend);
  };
  if (l.tend)
    return go(k_step<PMix, true>, k_step<PMix, true, false, false, true>,
              k_step<PMix, true, false, false, false, kBlock / 2>);
  if (line)
    return go(k_step<PMix, false, false, true>, k_step<PMix, false, false, true, true>, k_step<PMix, false, false, true>);
  return go(k_step<PMix, false>, k_step<PMix, false, false, false, true>,
            k_step<PMix, false, false, false, false, kBlock / 2>);
}

}  // namespace casim_dev
