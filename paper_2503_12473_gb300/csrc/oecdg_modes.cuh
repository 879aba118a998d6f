// oecdg_modes.cuh -- mode lists of the 2D spaces Q^k and P^k, field counts and the
// quadrature rules of runtime point loops, for the degree-generic 2D kernels.
#pragma once

#include "oecdg_poly.cuh"

namespace oecdg {

// Mode lists.  Q^k: index b (k+1) + a.  P^k: by total degree s = a + b, then
// by decreasing a (index of (a, b) = s (s+1) / 2 + b).  In closed form (k <= 3):
// nvcc does not fold a recursive function of an unrolled loop's index, the arrays
// of modes then go to local memory with computed indices, and in the Burgers P^k
// stage it (13.0) gave the x part's and the y part's array one slot there.
__host__ __device__ constexpr int pk_degree(int m) { return (m >= 1) + (m >= 3) + (m >= 6); }
__host__ __device__ constexpr int pk_b(int m) { return m - pk_degree(m) * (pk_degree(m) + 1) / 2; }
__host__ __device__ constexpr int pk_a(int m) { return pk_degree(m) - pk_b(m); }

template <int K, int B>
struct Modes2 {
  static constexpr int M = B == BASIS_Q ? (K + 1) * (K + 1) : (K + 1) * (K + 2) / 2;
  __host__ __device__ static constexpr int a(int m) { return B == BASIS_Q ? m % (K + 1) : pk_a(m); }
  __host__ __device__ static constexpr int b(int m) { return B == BASIS_Q ? m / (K + 1) : pk_b(m); }
  // phi_m and its reference derivatives (dx, dy) at (x, y)
  __host__ __device__ static constexpr double phi(int m, int dx, int dy, double x, double y) {
    return lpd(a(m), dx, x) * lpd(b(m), dy, y);
  }
};

template <int SYS>
struct Fields2 {
  static constexpr int F = SYS == SYS_EULER ? 4 : 1;
};

// Gauss nodes and weights of the N-point rules (N = 2, 3, 4) for runtime
// point loops: [N - 2][q].
static __constant__ double GNK[3][4] = {{gn1(2, 0), gn1(2, 1), 0.0, 0.0},
                                 {gn1(3, 0), gn1(3, 1), gn1(3, 2), 0.0},
                                 {gn1(4, 0), gn1(4, 1), gn1(4, 2), gn1(4, 3)}};
static __constant__ double GWK[3][4] = {{gw1(2, 0), gw1(2, 1), 0.0, 0.0},
                                 {gw1(3, 0), gw1(3, 1), gw1(3, 2), 0.0},
                                 {gw1(4, 0), gw1(4, 1), gw1(4, 2), gw1(4, 3)}};

}  // namespace oecdg
