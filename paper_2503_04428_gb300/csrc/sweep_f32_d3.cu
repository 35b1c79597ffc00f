// Fused sweep kernels: float state, 3D grids with the exact Riemann solver (all scalar counts).
#include "sweep.cuh"

namespace hydro {
HYDRO_SWEEP_DISPATCH_EXACT(float, 3)
}  // namespace hydro
