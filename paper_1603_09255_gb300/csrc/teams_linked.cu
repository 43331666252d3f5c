// Team kernel of members with a linkage map.
#include "generations.cuh"

namespace spg {

SoloKernel team_kernel_linked() { return team_instance<true, false, true>(); }

}  // namespace spg
