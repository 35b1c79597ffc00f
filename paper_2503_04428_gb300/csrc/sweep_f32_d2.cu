// Fused sweep kernels: float state, 2D grids with the exact Riemann solver (all scalar counts).
#include "sweep.cuh"

namespace hydro {
HYDRO_SWEEP_DISPATCH_EXACT(float, 2)
}  // namespace hydro
