// Pass 2 of the forward: the instantiations of the FWM grids.
#include "kint_fwd_main.cuh"

namespace kint {

cudaError_t launch_fwd_main_fwm(const Maps& maps, const Params& p, int smem_bytes, cudaStream_t s, const Sched& sch) {
  return p.calib == CAL_FWMR ? launch_main_grid<CAL_FWMR>(maps, p, smem_bytes, s, sch)
                             : launch_main_grid<CAL_FWM>(maps, p, smem_bytes, s, sch);
}

}  // namespace kint
