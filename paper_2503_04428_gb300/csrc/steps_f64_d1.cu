// Several steps of small 1D grids in one launch: double state.
#include "sweep.cuh"

namespace hydro {
HYDRO_STEPS_DISPATCH(double, 1, HYDRO_RS_ALL)
}  // namespace hydro
