// oecdg_2dk_delta.cu -- the 2D damping coefficients as a result.
#include "oecdg_oe2k.cuh"

namespace oecdg {

cudaError_t launch_delta2k(int sys, int bc, int k, int basis, const Geo& g, const double* uh, double* delta,
                           const double* dt, const double* sigma, int* status, cudaStream_t st) {
  return oe2k<OEK_DELTA>(sys, bc, k, basis, g, uh, delta, dt, sigma, status, st);
}

}  // namespace oecdg
