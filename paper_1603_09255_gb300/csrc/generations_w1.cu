// Generation kernel instances for L = 32 loci (W = 1).
#include "generations.cuh"

namespace spg {

SoloKernel solo_kernel_w1(bool linked, bool weighted) {
    if (linked) return weighted ? solo_instance<1, true, true>() : solo_instance<1, true, false>();
    return weighted ? solo_instance<1, false, true>() : solo_instance<1, false, false>();
}

}  // namespace spg
