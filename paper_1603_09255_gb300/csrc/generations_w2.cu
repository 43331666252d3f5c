// Generation kernel instances for L = 64 loci (W = 2).
#include "generations.cuh"

namespace spg {

SoloKernel solo_kernel_w2(bool linked, bool weighted) {
    if (linked) return weighted ? solo_instance<2, true, true>() : solo_instance<2, true, false>();
    return weighted ? solo_instance<2, false, true>() : solo_instance<2, false, false>();
}

}  // namespace spg
