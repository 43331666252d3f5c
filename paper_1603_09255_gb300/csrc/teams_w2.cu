// Team kernel instances for L = 64 loci (W = 2).
#include "generations.cuh"

namespace spg {

SoloKernel team_kernel_w2(uint32_t kind) { return team_kernel_of<2>(kind); }

}  // namespace spg
