// k_cu2d_f32_star_r57.cu -- instantiations of the CUDA-core sweep launchers: 2-D FP32 star, r = 5..7.
#include "k_cuda_core_impl.cuh"

namespace gbs {

stencil_status launch_cu2d_f32_star_r57(const Plan &p, const void *in, void *out, int t, cudaStream_t st)
{
    return cuimpl::launch2d_range<float, 1, 5, 7>(p, in, out, t, st);
}

}  // namespace gbs
