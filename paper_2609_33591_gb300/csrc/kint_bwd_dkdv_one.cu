// dK/dV kernels of the backward (App. B): the one-product instantiations (d = 128, 3xTF32).
#include "kint_bwd_kv.cuh"

namespace kint {

template cudaError_t launch_bwd_dkdv_t<false, DKV_DV>(const Maps&, const Params&, int, cudaStream_t, const SnakeOrder&);
template cudaError_t launch_bwd_dkdv_t<false, DKV_DK>(const Maps&, const Params&, int, cudaStream_t, const Sched&);

}  // namespace kint
