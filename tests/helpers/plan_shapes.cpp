// The planner of the walkers' launches (wl_plan.h) as a shared library, for a GPU that is
// given by its limits: blocks of an SM by shared memory, and by what the registers of the
// two kernels leave room for.
#include "../../paper_1302_2320_gb300/csrc/wl_plan.h"

using namespace wl;
using namespace wl::rt;

extern "C" int turns_of(const Shape* sh, long long running, long long moves) { return line_turns(*sh, running, moves); }

extern "C" int plan_shapes(const ShapeKey* k, const Gpu* gpu, int max_lone, int max_batch, Shape* out)
{
    auto resident = [&](const Slot& slot, size_t smem, int) {
        const size_t block = (smem + (size_t)gpu->reserved + 127) / 128 * 128;
        return std::min((int)((size_t)gpu->per_sm / block), slot.lone ? max_lone : max_batch);
    };
    return (int)plan_shape(*k, *gpu, resident, out);
}
