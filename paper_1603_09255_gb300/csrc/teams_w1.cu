// Team kernel instances for L = 32 loci (W = 1).
#include "generations.cuh"

namespace spg {

SoloKernel team_kernel_w1(uint32_t kind) { return team_kernel_of<1>(kind); }

}  // namespace spg
