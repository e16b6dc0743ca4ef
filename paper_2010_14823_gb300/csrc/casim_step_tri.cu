// The triple-moment step kernels.
#include "casim_step_impl.cuh"

namespace casim_dev {
template struct StepKernels<PolicyMix3, PolicyF643>;
}  // namespace casim_dev
