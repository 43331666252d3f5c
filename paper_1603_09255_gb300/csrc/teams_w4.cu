// Team kernel instances for L = 128 loci (W = 4).
#include "generations.cuh"

namespace spg {

SoloKernel team_kernel_w4(uint32_t kind) { return team_kernel_of<4>(kind); }

}  // namespace spg
