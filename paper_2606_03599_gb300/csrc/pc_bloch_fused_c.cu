// Fused preconditioner kernels (pc_bloch_fused.cuh), part c of the sizes.
#include "pc_bloch_fused.cuh"

namespace pc {
namespace fused {
PC_FUSED_TU(launch_c, PC_FUSED_C)
}  // namespace fused
}  // namespace pc
