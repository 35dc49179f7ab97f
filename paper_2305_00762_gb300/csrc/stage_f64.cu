// FP64 instantiation of the fused stage kernel (the plain method).
#include "fixed_stage.cuh"

namespace gbr {

// 16 x 16 tiles of 288 threads, two CTAs per SM: the tile's 544 faces are 17
// warps of work, two rounds of nine warps (256 threads need three, the last
// with one warp busy: 1024^2 step 1.57 -> 1.44 ms, viscous 1280 x 640 2.46 ->
// 2.28 ms, at 96 registers instead of 128).
cudaError_t launch_stage_f64(const StageParams& p, cudaStream_t s)
{
    if (p.ph.cons) return launch_stage_cons_f64(p, s);
    if (p.ph.order == 4) {
        if (p.ph.mu > 0.0) return launch_fixed<16, 16, 288, true, 4>(p, s);
        return launch_fixed<16, 16, 288, false, 4>(p, s);
    }
    if (p.ph.mu > 0.0) return launch_fixed<16, 16, 288, true, 7>(p, s);
    return launch_fixed<16, 16, 288, false, 7>(p, s);
}

}  // namespace gbr
