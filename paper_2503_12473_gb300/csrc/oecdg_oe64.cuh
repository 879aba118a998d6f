// oecdg_oe64.cuh -- the OE step's sums over a quarter's half-faces in FP64
// (arXiv:2503.12473, Section 2.2), for the damping coefficients as a result.
//
// The fixed-point sums of the OE kernels cut every derivative at about 2^-53 of the
// cell's local variation: enough for the decay, since sigma is at least that variation's
// size, but a coefficient by itself can be far below it (third derivatives of smooth data:
// P^3 on a wave over 128 cells has delta^3 to 1e-11 from the fixed-point sums, to 2e-16
// from these).  The FP64 pipe sets their time, as it did the OE step's before the
// fixed-point sums: a launch takes 2.30 ms on P^3 Euler 256^2 (2.4 there) where the step takes
// 0.34, 6.1 on Q^2 512^2 (0.62).
#pragma once

#include "oecdg_common.cuh"
#include "oecdg_modes.cuh"

namespace oecdg {

// The power of two that brings a field's coefficients to the size of its sigma (isg =
// 1 / sigma), so that no square leaves the range of a double; 1 for a constant field.
__device__ __forceinline__ double oe_unit(double isg) {
  const int hi = __double2hiint(isg) & 0x7ff00000;
  return hi == 0 || hi == 0x7ff00000 ? 1.0 : __hiloint2double(hi, 0);
}

// S[n (K+1) + m]: over the N = K+1 points of the quarter's half-face normal to
// direction n, the rule's sum of the order-m norm of K's trace minus the overlapping
// cell, in units of (2 / min(hx, hy))^m / unit.  us, uo: mode 0 of K's and of the
// overlapping cell's field (stride P per mode).  flip: bits 0, 1 the quarter (sx, sy),
// bits 2, 3 the overlapping cell is a mirror image across a wall normal to x, y, bit 4
// its field changes sign there.  In coordinates mirrored so that the quarter is K's low
// half: K's face at -1, the overlapping cell's centre line at 0, zeta' = zeta + 1.
template <int K, int B>
static __device__ __noinline__ void oe_quarter_fp64(const double* __restrict__ us, const double* __restrict__ uo,
                                                    long long P, unsigned flip, double unit, double i2x, double i2y,
                                                    double* __restrict__ S) {
  using MD = Modes2<K, B>;
  constexpr int M = MD::M, N = K + 1;
  const double rx = i2x < i2y ? i2x / i2y : 1.0, ry = i2y < i2x ? i2y / i2x : 1.0;
  double k[M], o[M];
#pragma unroll
  for (int m = 0; m < M; ++m) {
    const unsigned fk = (MD::a(m) & 1 ? flip : 0u) ^ (MD::b(m) & 1 ? flip >> 1 : 0u);
    const unsigned fo = fk ^ (MD::a(m) & 1 ? flip >> 2 : 0u) ^ (MD::b(m) & 1 ? flip >> 3 : 0u) ^ (flip >> 4);
    k[m] = us[m * P];
    o[m] = uo[m * P];
    if (fk & 1) k[m] = -k[m];
    if (fo & 1) o[m] = -o[m];
  }
  o[0] -= k[0];  // the means enter by their difference
  k[0] = 0.0;
#pragma unroll
  for (int m = 0; m < M; ++m) {
    k[m] *= unit;
    o[m] *= unit;
  }
#pragma unroll
  for (int n = 0; n < 2; ++n) {
    // E[an][at]: coefficient of P_at(zeta) in the difference's an-th normal derivative
    double E[K + 1][K + 1], W[K + 1][K + 1];
#pragma unroll
    for (int d = 0; d <= K; ++d)
#pragma unroll
      for (int a = 0; a <= K; ++a) E[d][a] = W[d][a] = 0.0;
#pragma unroll
    for (int m = 0; m < M; ++m) {
      const int an = n == 0 ? MD::a(m) : MD::b(m), at = n == 0 ? MD::b(m) : MD::a(m);
#pragma unroll
      for (int d = 0; d <= an; ++d) {
        E[d][at] = fma(lpd(an, d, -1.0), k[m], E[d][at]);
        if (lpd(an, d, 0.0) != 0.0) W[d][at] = fma(lpd(an, d, 0.0), o[m], W[d][at]);
      }
    }
#pragma unroll
    for (int d = 0; d <= K; ++d)
#pragma unroll
      for (int a = 0; a <= K; ++a) {
        double e = E[d][a] - W[d][a];
#pragma unroll
        for (int b = a + 1; b <= K; ++b)
          if (!(B == BASIS_P && b + d > K)) e = fma(-lshift(b, a, 1.0), W[d][b], e);
        E[d][a] = e;
      }
    const double sn = n == 0 ? rx : ry, st = n == 0 ? ry : rx;
    double pn = 1.0, pt[K + 1];
    pt[0] = 1.0;
#pragma unroll
    for (int d = 1; d <= K; ++d) {
      pn *= sn;
      pt[d] = pt[d - 1] * st;
#pragma unroll
      for (int a = 0; a <= K; ++a) E[d][a] *= pn;
    }
    double s[K + 1];
#pragma unroll
    for (int m = 0; m <= K; ++m) s[m] = 0.0;
#pragma unroll
    for (int q = 0; q < N; ++q) {
      const double wq = gw1(N, q), t = 0.5 * gn1(N, q) - 0.5;
#pragma unroll
      for (int m = 0; m <= K; ++m) {
        double ss = 0.0;
#pragma unroll
        for (int an = 0; an <= m; ++an) {
          const int at = m - an;
          double v = 0.0;
#pragma unroll
          for (int a = at; a <= K; ++a)
            if (!(B == BASIS_P && a + an > K)) v = fma(E[an][a], lpd(a, at, t), v);
          if (at > 0) v *= pt[at];
          ss = fma(v, v, ss);
        }
        // sums below 2^-1022 are far below the unit
        if (__double2hiint(ss) >= 0x00100000) s[m] = fma(wq, sqrt_pos(ss), s[m]);
      }
    }
#pragma unroll
    for (int m = 0; m <= K; ++m) S[n * (K + 1) + m] = s[m];
  }
}

}  // namespace oecdg
