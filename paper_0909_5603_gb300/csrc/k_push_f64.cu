// k_push_f64.cu -- double instantiations of the fused particle kernel, without an injection plane.
#include "k_push.cuh"

namespace pic {

cudaError_t dispatch_particles_f64(int ndim, int order, int pusher, const Launch *L, const OneInst *one, size_t smem,
                                     cudaStream_t s)
{
    return dispatch_particles_t<double, false>(ndim, order, pusher, L, one, smem, s);
}

}  // namespace pic
