// Generation kernel instances for L = 128 loci (W = 4).
#include "generations.cuh"

namespace spg {

SoloKernel solo_kernel_w4(bool linked, bool weighted) {
    if (linked) return weighted ? solo_instance<4, true, true>() : solo_instance<4, true, false>();
    return weighted ? solo_instance<4, false, true>() : solo_instance<4, false, false>();
}

}  // namespace spg
