// Instantiations of the line pass kernel (lines_kernel.cuh) for m = 1 (tau plays no part):
// the diagonal pass (also for a full sweep of LINE_KMAX thresholds) and the
// vertical pass.  One group per translation unit, so they compile in parallel.
#include "lines_kernel.cuh"

namespace rqa {

LinesKernel lines_kernel_m1t1(bool vert, bool full)
{
    if (vert) return k_lines<1, 1, true>;
    return full ? k_lines<1, 1, false, true> : k_lines<1, 1, false>;
}

}  // namespace rqa
