// dK/dV kernels of the backward (App. B): the instantiations with both products, and the launch
// entry that picks an instantiation.
#include "kint_bwd_kv.cuh"

namespace kint {

template cudaError_t launch_bwd_dkdv_t<false, DKV_BOTH>(const Maps&, const Params&, int, cudaStream_t, const SnakeOrder&);

cudaError_t launch_bwd_dkdv(const Maps& maps, const Params& p, int smem_bytes, cudaStream_t s, const Sched& sch) {
  if (p.dkv_sel == DKV_DV) return launch_bwd_dkdv_t<false, DKV_DV>(maps, p, smem_bytes, s, SnakeOrder{});  // (dS is not formed)
  const bool rs = p.dsum_out || p.dabs_out;
  if (p.dkv_sel == DKV_DK)
    return rs ? launch_bwd_dkdv_t<true, DKV_DK>(maps, p, smem_bytes, s, sch)
              : launch_bwd_dkdv_t<false, DKV_DK>(maps, p, smem_bytes, s, sch);
  return rs ? launch_bwd_dkdv_t<true, DKV_BOTH>(maps, p, smem_bytes, s, SnakeOrder{})
            : launch_bwd_dkdv_t<false, DKV_BOTH>(maps, p, smem_bytes, s, SnakeOrder{});
}

}  // namespace kint
