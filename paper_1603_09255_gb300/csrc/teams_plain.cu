// Team kernel of plain members.
#include "generations.cuh"

namespace spg {

SoloKernel team_kernel_plain() { return team_instance<false, false, false>(); }

}  // namespace spg
