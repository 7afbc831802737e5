// ccmc_step_generic_f32.cu -- the step kernels for a generic Hamiltonian with FP32 matrix elements.
#include "ccmc_kernels.cuh"

namespace ccmc {

template cudaError_t launch_phases<float, false>(const StepArgs *, int, int, const Shapes &, bool, cudaStream_t, i64 *,
                                               const cudaEvent_t *, const FlatPlan *);

}  // namespace ccmc
