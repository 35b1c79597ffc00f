// Several steps of small 2D grids in one launch: float state.
#include "sweep.cuh"

namespace hydro {
HYDRO_STEPS_DISPATCH(float, 2, HYDRO_RS_EXACT_ONLY)
}  // namespace hydro
