// Fused kernel, two atoms per warp: floating-point scatter, tables in global memory (see the end of megakernel.cuh).
#include "megakernel.cuh"

namespace mlip {

MegaKernel mega_two(bool list16) { return list16 ? k_mega<2, true, true, false, true> : k_mega<2, true, true, false, false>; }
MegaKernel mega_two_global(bool det, bool list16) {
    static const MegaKernel kernels[4] = {k_mega<2, true, false, false, false>, k_mega<2, true, false, false, true>, k_mega<2, true, false, true, false>, k_mega<2, true, false, true, true>};
    return kernels[(det ? 2 : 0) + (list16 ? 1 : 0)];
}

}  // namespace mlip
