// wl_lone.cu -- instantiations and dispatch of the block-per-line walker.
#include <type_traits>

#include "wl_launch.cuh"
#include "wl_lone.cuh"

namespace wl {

cudaError_t launch_lone(bool det, dim3 grid, dim3 block, size_t smem, cudaStream_t s, const WalkArgs& a, int* bps)
{
    const bool tri = a.g.shape == kShapeTriangular;
    auto pick = [&](auto word) {
        constexpr int W = decltype(word)::value;
        return tri ? (det ? lone_kernel<true, true, W> : lone_kernel<true, false, W>)
                   : (det ? lone_kernel<false, true, W> : lone_kernel<false, false, W>);
    };
    auto* fn = a.lone == 4 ? pick(std::integral_constant<int, 4>{}) : pick(std::integral_constant<int, 1>{});
    return launch_or_query(fn, grid, block, smem, s, a, bps);
}

}  // namespace wl
