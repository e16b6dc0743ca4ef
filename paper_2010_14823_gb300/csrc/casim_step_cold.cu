// The standard configuration's step kernels.
#include "casim_step_impl.cuh"

namespace casim_dev {
template struct StepKernels<PolicyMix, PolicyF64>;
}  // namespace casim_dev
