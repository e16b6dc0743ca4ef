// The warm configuration's step kernels with aerosol mass and with triple-moment rain.
#include "casim_step_impl.cuh"

namespace casim_dev {
template struct StepKernels<PolicyMixWarmAero, PolicyF64WarmAero>;
template struct StepKernels<PolicyMixWarm3, PolicyF64Warm3>;
}  // namespace casim_dev
