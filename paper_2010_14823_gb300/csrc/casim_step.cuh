// Launch of the step kernels.  Each configuration's kernels are compiled in a
// translation unit of their own (casim_step_*.cu), side by side.
#pragma once

#include "casim_device.cuh"

namespace casim_dev {

struct StepLaunch {
  bool mixed;
  bool line;             // the state is mapped host memory (the mixed step's whole-line stores)
  int nsm;
  cudaStream_t stream;
  double *tend;          // the source-term mode's output, or null: the in-place step
};

// the kernels of one configuration, mixed and FP64
template <class PMix, class PF64>
struct StepKernels {
  // a staged step kernel may use the dynamic shared memory of a column of the
  // largest level count
  static cudaError_t allow_smem();
  static cudaError_t launch(const StepLaunch &l, const KArgs &a, const KParams &kp);
};

using StepCold = StepKernels<PolicyMix, PolicyF64>;
using StepWarm = StepKernels<PolicyMixWarm, PolicyF64Warm>;
using StepWarmAero = StepKernels<PolicyMixWarmAero, PolicyF64WarmAero>;
using StepWarm3 = StepKernels<PolicyMixWarm3, PolicyF64Warm3>;
using StepAero = StepKernels<PolicyMixAero, PolicyF64Aero>;
using Step3 = StepKernels<PolicyMix3, PolicyF643>;

extern template struct StepKernels<PolicyMix, PolicyF64>;
extern template struct StepKernels<PolicyMixWarm, PolicyF64Warm>;
extern template struct StepKernels<PolicyMixWarmAero, PolicyF64WarmAero>;
extern template struct StepKernels<PolicyMixWarm3, PolicyF64Warm3>;
extern template struct StepKernels<PolicyMixAero, PolicyF64Aero>;
extern template struct StepKernels<PolicyMix3, PolicyF643>;

}  // namespace casim_dev
