// Team kernel of members with dominance, large effects or a large bias.
#include "generations.cuh"

namespace spg {

SoloKernel team_kernel_general() { return team_instance<false, false, true>(); }

}  // namespace spg
