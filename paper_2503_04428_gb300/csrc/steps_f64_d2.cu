// Several steps of small 2D grids in one launch: double state.
#include "sweep.cuh"

namespace hydro {
HYDRO_STEPS_DISPATCH(double, 2, HYDRO_RS_ALL)
}  // namespace hydro
