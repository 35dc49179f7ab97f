// FP64 form: the seventh-order inviscid instances, and the choice among the
// others (viscous, fourth-order, MEG7-cons: a translation unit each).
#include "fixed_stage.cuh"

namespace gbr {

cudaError_t stage_f64_maps_ghosts(const Grid& g, const Physics& ph, bool* maps)
{
    TileShape t;
    const cudaError_t e = fixed_tile_shape(g, ph.cons != 0, ph.mu > 0.0, &t);
    if (e == cudaSuccess) *maps = fixed_maps_ghosts(t.bx);
    return e;
}

cudaError_t launch_stage_f64(const StageParams& p, cudaStream_t s)
{
    // (with a stage update the kernel holds -dt Res in the residual's place: finish_tile)
    if (p.res && p.qout) return cudaErrorInvalidValue;
    if (p.ph.cons) return launch_stage_cons_f64(p, s);
    if (p.ph.order == 4) return launch_stage_order4_f64(p, s);
    if (p.ph.mu > 0.0) return launch_stage_viscous_f64(p, s);
    return launch_fixed<false, 7>(p, s);
}

}  // namespace gbr
