// Generation kernel instances for L = 64 loci (W = 2).
#include "generations.cuh"

namespace spg {

SoloKernel solo_kernel_w2(bool linked, bool weighted, bool general) {
    if (linked) return weighted ? solo_instance<2, true, true>(general) : solo_instance<2, true, false>(general);
    return weighted ? solo_instance<2, false, true>(general) : solo_instance<2, false, false>(general);
}

}  // namespace spg
