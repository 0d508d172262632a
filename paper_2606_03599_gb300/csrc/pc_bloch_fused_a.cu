// Fused preconditioner kernels (pc_bloch_fused.cuh), part a of the sizes.
#include "pc_bloch_fused.cuh"

namespace pc {
namespace fused {
PC_FUSED_TU(launch_a, PC_FUSED_A)
}  // namespace fused
}  // namespace pc
