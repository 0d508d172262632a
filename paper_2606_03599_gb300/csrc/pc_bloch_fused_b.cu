// Fused preconditioner kernels (pc_bloch_fused.cuh), part b of the sizes.
#include "pc_bloch_fused.cuh"

namespace pc {
namespace fused {
PC_FUSED_TU(launch_b, PC_FUSED_B)
}  // namespace fused
}  // namespace pc
