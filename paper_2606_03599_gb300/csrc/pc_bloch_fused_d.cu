// Fused preconditioner kernels (pc_bloch_fused.cuh), part d of the sizes.
#include "pc_bloch_fused.cuh"

namespace pc {
namespace fused {
PC_FUSED_TU(launch_d, PC_FUSED_D)
}  // namespace fused
}  // namespace pc
