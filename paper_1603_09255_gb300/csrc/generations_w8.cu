// Generation kernel instances for L = 256 loci (W = 8).
#include "generations.cuh"

namespace spg {

SoloKernel solo_kernel_w8(bool linked, bool weighted, bool general) {
    if (linked) return weighted ? solo_instance<8, true, true>(general) : solo_instance<8, true, false>(general);
    return weighted ? solo_instance<8, false, true>(general) : solo_instance<8, false, false>(general);
}

}  // namespace spg
