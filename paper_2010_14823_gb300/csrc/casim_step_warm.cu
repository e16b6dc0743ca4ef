// The warm configuration's step kernels.
#include "casim_step_impl.cuh"

namespace casim_dev {
template struct StepKernels<PolicyMixWarm, PolicyF64Warm>;
}  // namespace casim_dev
