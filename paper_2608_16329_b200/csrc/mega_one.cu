// Fused kernel, one atom per warp; two with the integer scatter (see the end of megakernel.cuh).
#include "megakernel.cuh"

namespace mlip {

MegaKernel mega_one(bool det, bool list16) {
    static const MegaKernel kernels[4] = {k_mega<1, false, true, false, false>, k_mega<1, false, true, false, true>, k_mega<1, false, true, true, false>, k_mega<1, false, true, true, true>};
    return kernels[(det ? 2 : 0) + (list16 ? 1 : 0)];
}
MegaKernel mega_two_fixed(bool list16) { return list16 ? k_mega<2, true, true, true, true> : k_mega<2, true, true, true, false>; }

}  // namespace mlip
