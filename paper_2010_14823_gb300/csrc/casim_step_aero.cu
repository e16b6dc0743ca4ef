// The step kernels with activated-aerosol mass.
#include "casim_step_impl.cuh"

namespace casim_dev {
template struct StepKernels<PolicyMixAero, PolicyF64Aero>;
}  // namespace casim_dev
