// Team kernel instances for L = 256 loci (W = 8).
#include "generations.cuh"

namespace spg {

SoloKernel team_kernel_w8(uint32_t kind) { return team_kernel_of<8>(kind); }

}  // namespace spg
