// FP64 form, the fourth-order member of the scheme's family.
#include "fixed_stage.cuh"

namespace gbr {

cudaError_t launch_stage_order4_f64(const StageParams& p, cudaStream_t s)
{
    if (p.ph.mu > 0.0) return launch_fixed<true, 4>(p, s);
    return launch_fixed<false, 4>(p, s);
}

}  // namespace gbr
