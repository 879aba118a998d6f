// oecdg_2dk_oe.cu -- the OE step of the degree-generic 2D kernels on square cells.
#include "oecdg_oe2k.cuh"

namespace oecdg {

cudaError_t launch_oe2k(int sys, int bc, int k, int basis, const Geo& g, const double* uh, double* usig,
                        const double* dt, const double* sigma, int* status, cudaStream_t st) {
  return g.hx == g.hy ? oe2k<OEK_SQUARE>(sys, bc, k, basis, g, uh, usig, dt, sigma, status, st)
                      : launch_oe2k_oblong(sys, bc, k, basis, g, uh, usig, dt, sigma, status, st);
}

}  // namespace oecdg
