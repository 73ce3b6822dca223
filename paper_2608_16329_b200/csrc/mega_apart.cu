// Fused kernel, two atoms per warp, one after the other.
#include "megakernel.cuh"

namespace mlip {

MegaKernel mega_apart(bool in_smem, bool det, bool list16) {
    static const MegaKernel kernels[8] = {k_mega<2, false, false, false, false>, k_mega<2, false, false, false, true>, k_mega<2, false, false, true, false>, k_mega<2, false, false, true, true>,
                                          k_mega<2, false, true, false, false>, k_mega<2, false, true, false, true>, k_mega<2, false, true, true, false>, k_mega<2, false, true, true, true>};
    return kernels[(in_smem ? 4 : 0) + (det ? 2 : 0) + (list16 ? 1 : 0)];
}

}  // namespace mlip
