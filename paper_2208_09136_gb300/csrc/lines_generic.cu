// Instantiations of the line pass kernel (lines_kernel.cuh) for the other
// embeddings: compile-time m with the delay read at run time (any tau), and
// the fully generic one (m and tau at run time).
#include "lines_kernel.cuh"

namespace rqa {

LinesKernel lines_kernel_generic(int m, bool vert)
{
    switch (m) {
    case 2: return vert ? k_lines<2, 0, true> : k_lines<2, 0, false>;
    case 3: return vert ? k_lines<3, 0, true> : k_lines<3, 0, false>;
    case 4: return vert ? k_lines<4, 0, true> : k_lines<4, 0, false>;
    default: return vert ? k_lines<0, 0, true> : k_lines<0, 0, false>;
    }
}

}  // namespace rqa
