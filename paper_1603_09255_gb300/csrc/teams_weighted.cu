// Team kernel of members with parent weights.
#include "generations.cuh"

namespace spg {

SoloKernel team_kernel_weighted() { return team_instance<false, true, true>(); }

}  // namespace spg
