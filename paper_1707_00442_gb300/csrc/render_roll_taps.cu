// render_roll_taps.cu -- the rolling marcher's instances for the per-axis taps (Algorithm 9).
#include "render_roll.cuh"

namespace shw {

shw_status render_roll_taps(int mode, int interp, const shw_volume &v, const shw_camera &cam, const RenderArgs &a,
                            cudaStream_t st)
{
    if (interp != SHW_TRILINEAR || v.storage != SHW_F32 || debug(SHW_DEBUG_NO_STAGING)) return SHW_EUNSUPPORTED;
    if ((long long)v.nx * v.ny * v.nz >= (1LL << 31)) return SHW_EUNSUPPORTED;
    return roll_launch<kRollTaps>(mode, v, cam, a, st);
}

}  // namespace shw
