// Several steps of small 1D grids in one launch: float state.
#include "sweep.cuh"

namespace hydro {
HYDRO_STEPS_DISPATCH(float, 1, HYDRO_RS_ALL)
}  // namespace hydro
