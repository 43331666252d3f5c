// Generation kernel instances for L = 256 loci (W = 8).
#include "generations.cuh"

namespace spg {

SoloKernel solo_kernel_w8(bool linked, bool weighted) {
    if (linked) return weighted ? solo_instance<8, true, true>() : solo_instance<8, true, false>();
    return weighted ? solo_instance<8, false, true>() : solo_instance<8, false, false>();
}

}  // namespace spg
