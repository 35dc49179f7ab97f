// FP64 form, MEG7-cons (conservative-variable reconstruction, seventh order).
#include "fixed_stage.cuh"

namespace gbr {

cudaError_t launch_stage_cons_f64(const StageParams& p, cudaStream_t s)
{
    if (p.ph.mu > 0.0) return launch_fixed<true, 7, true>(p, s);
    return launch_fixed<false, 7, true>(p, s);
}

}  // namespace gbr
