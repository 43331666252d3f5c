// Generation kernel instances for L = 32 loci (W = 1).
#include "generations.cuh"

namespace spg {

SoloKernel solo_kernel_w1(bool linked, bool weighted, bool general) {
    if (linked) return weighted ? solo_instance<1, true, true>(general) : solo_instance<1, true, false>(general);
    return weighted ? solo_instance<1, false, true>(general) : solo_instance<1, false, false>(general);
}

}  // namespace spg
