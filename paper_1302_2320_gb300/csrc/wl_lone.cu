// wl_lone.cu -- instantiations and dispatch of the block-per-line walker.
#include "wl_launch.cuh"
#include "wl_lone.cuh"

namespace wl {

cudaError_t launch_lone(bool det, dim3 grid, dim3 block, size_t smem, cudaStream_t s, const WalkArgs& a, int* bps)
{
    auto* fn = a.g.shape == kShapeTriangular ? (det ? lone_kernel<true, true> : lone_kernel<true, false>)
                                             : (det ? lone_kernel<false, true> : lone_kernel<false, false>);
    return launch_or_query(fn, grid, block, smem, s, a, bps);
}

}  // namespace wl
