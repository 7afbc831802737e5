// ccmc_step_generic_f64.cu -- the step kernels for a generic Hamiltonian with FP64 matrix elements.
#include "ccmc_kernels.cuh"

namespace ccmc {

template cudaError_t launch_phases<double, false>(const StepArgs *, int, int, const Shapes &, bool, cudaStream_t, i64 *,
                                               const cudaEvent_t *, const FlatPlan *);

}  // namespace ccmc
