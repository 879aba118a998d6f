// oecdg_2dk_oblong.cu -- the OE step of the degree-generic 2D kernels on cells that are not square.
#include "oecdg_oe2k.cuh"

namespace oecdg {

cudaError_t launch_oe2k_oblong(int sys, int bc, int k, int basis, const Geo& g, const double* uh, double* usig,
                               const double* dt, const double* sigma, int* status, cudaStream_t st) {
  return oe2k<OEK_OBLONG>(sys, bc, k, basis, g, uh, usig, dt, sigma, status, st);
}

}  // namespace oecdg
