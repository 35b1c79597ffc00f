// Fused sweep kernels: float state, 3D grids (all solvers and scalar counts).
#include "sweep.cuh"

namespace hydro {
HYDRO_SWEEP_DISPATCH(float, 3)
}  // namespace hydro
