// ccmc_step_gas_f32.cu -- the step kernels for the electron gas with FP32 matrix elements.
#include "ccmc_kernels.cuh"

namespace ccmc {

template cudaError_t launch_phases<float, true>(const StepArgs *, int, int, const Shapes &, bool, cudaStream_t, i64 *,
                                               const cudaEvent_t *, const FlatPlan *);

}  // namespace ccmc
