// Team kernel of members with a linkage map and parent weights.
#include "generations.cuh"

namespace spg {

SoloKernel team_kernel_both() { return team_instance<true, true, true>(); }

}  // namespace spg
