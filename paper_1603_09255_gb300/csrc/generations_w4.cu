// Generation kernel instances for L = 128 loci (W = 4).
#include "generations.cuh"

namespace spg {

SoloKernel solo_kernel_w4(bool linked, bool weighted, bool general) {
    if (linked) return weighted ? solo_instance<4, true, true>(general) : solo_instance<4, true, false>(general);
    return weighted ? solo_instance<4, false, true>(general) : solo_instance<4, false, false>(general);
}

}  // namespace spg
