// FP32 storage, FP32 (packed f32x2) compute, all faces periodic: the step
// kernels that also write the periodic ghost images of their new cells.
#include "step_kernel.cuh"
#include "tiles.h"

namespace spfm {
cudaError_t launch_step_f32_img(const StepCoef<float> &c, const float *src, float *dst, int *err,
                                LaunchCfg cfg, TmaCache *tma, int which, cudaStream_t st)
{
    if (cfg.rounding == SPFM_ROUND_STOCHASTIC) return launch_step_f32_img_sr(c, src, dst, err, cfg, tma, which, st);
    const CUtensorMap *map = f32_step_map(tma, which, c, cfg.scheme, src);
    return launch_step_t<float, float, SPFM_F32_TX, SPFM_F32_TY, true, false, kSqTX, kSqTY>(
        c, src, dst, err, cfg, map, st);
}
}  // namespace spfm
