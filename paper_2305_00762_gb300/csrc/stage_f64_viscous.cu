// FP64 form, seventh order with the viscous terms.
#include "fixed_stage.cuh"

namespace gbr {

cudaError_t launch_stage_viscous_f64(const StageParams& p, cudaStream_t s) { return launch_fixed<true, 7>(p, s); }

}  // namespace gbr
