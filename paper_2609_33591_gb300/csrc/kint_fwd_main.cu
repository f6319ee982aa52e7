// Pass 2 of the forward: the instantiations of the MinMax grid and the exponentials, and
// the launch entry.
#include "kint_fwd_main.cuh"

namespace kint {

cudaError_t launch_fwd_main_fwm(const Maps& maps, const Params& p, int smem_bytes, cudaStream_t s, const Sched& sch);

cudaError_t launch_fwd_main(const Maps& maps, const Params& p, int smem_bytes, cudaStream_t s, const Sched& sch) {
  switch (p.calib) {
    case CAL_SOFTMAX: return launch_main_exp<CAL_SOFTMAX>(maps, p, smem_bytes, s, sch);
    case CAL_EXP8: return launch_main_exp<CAL_EXP8>(maps, p, smem_bytes, s, sch);
    case CAL_EXPB: return launch_main_exp<CAL_EXPB>(maps, p, smem_bytes, s, sch);
    case CAL_MINMAX: return launch_main_grid<CAL_MINMAX>(maps, p, smem_bytes, s, sch);
    default: return launch_fwd_main_fwm(maps, p, smem_bytes, s, sch);
  }
}

}  // namespace kint
