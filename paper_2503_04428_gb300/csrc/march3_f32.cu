// The FP32 3D step of the ideal gas with HLL and HLLC (march3.cuh).
#include "march3.cuh"

namespace hydro {
template <int NSX>
static cudaError_t dispatch(const SweepArgs<float>& a, int rs, cudaStream_t s, LaunchShape* sh) {
  if (a.spherical)
    return rs == RS_HLL ? launch_march3<NSX, RS_HLL, true>(a, s, sh)
                        : launch_march3<NSX, RS_HLLC, true>(a, s, sh);
  return rs == RS_HLL ? launch_march3<NSX, RS_HLL, false>(a, s, sh)
                      : launch_march3<NSX, RS_HLLC, false>(a, s, sh);
}

cudaError_t march3_dispatch(const SweepArgs<float>& a, int nsx, int rs, cudaStream_t s, LaunchShape* sh) {
  switch (nsx) {
    case 0: return dispatch<0>(a, rs, s, sh);
    case 1: return dispatch<1>(a, rs, s, sh);
    default: return dispatch<3>(a, rs, s, sh);
  }
}

bool march3_pays(const int* n, int nsx, int sms) {
  return nsx == 0 ? march3_pays<0>(n, sms) : nsx == 1 ? march3_pays<1>(n, sms) : march3_pays<3>(n, sms);
}
}  // namespace hydro
