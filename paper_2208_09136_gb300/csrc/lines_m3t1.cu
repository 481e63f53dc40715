// Instantiations of the line pass kernel (lines_kernel.cuh) for m = 3, tau = 1:
// the diagonal pass (also for a full sweep of LINE_KMAX thresholds) and the
// vertical pass.  One group per translation unit, so they compile in parallel.
#include "lines_kernel.cuh"

namespace rqa {

LinesKernel lines_kernel_m3t1(bool vert, bool full)
{
    if (vert) return k_lines<3, 1, true>;
    return full ? k_lines<3, 1, false, true> : k_lines<3, 1, false>;
}

}  // namespace rqa
