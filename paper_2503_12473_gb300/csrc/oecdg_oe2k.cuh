// oecdg_oe2k.cuh -- the OE step of the degree-generic 2D kernels (arXiv:2503.12473,
// Section 2.2).  Its three forms are translation units of their own (the build's time).
#pragma once

#include "oecdg_common.cuh"
#include "oecdg_fix.cuh"
#include "oecdg_kernels.h"
#include "oecdg_launch2k.h"
#include "oecdg_modes.cuh"
#include "oecdg_oe64.cuh"
#include "oecdg_oek.cuh"

namespace oecdg {

constexpr int NTK = 128;  // threads of an OE block: 4 rows of 8 cells, four lanes each

// The form of the sums: square cells, oblong ones (oecdg_oek.cuh), or FP64 ones for the
// coefficients as a result (oecdg_oe64.cuh), which write delta in place of the damped state.
enum { OEK_SQUARE = 0, OEK_OBLONG = 1, OEK_DELTA = 2 };
//
// Measured, a launch on square cells: P^3 Euler 256^2 0.34 ms (ALU pipe 60%), P^2 advection
// 512^2 0.20 ms (FP64 pipe 83%); the one-thread-per-cell FP64 form took about 2.4 and 1.1
// ms; OEK_DELTA takes 2.30 and 1.24.
struct OeK {
  double c[2][4];  // [direction][order]: the factor of the integer sums in delta^m
};

// delta_K^m, m = 0..K (Section 2.2): for every face e of K (x-faces: h_e = hx,
// beta_x; y-faces: h_e = hy, beta_y), over its 2 halves with K+1 Gauss points
// each, the integral of (sum_{|alpha| = m} (d^alpha (u_K - w))^2)^(1/2) with
// K's interior trace and the overlapping cell's solution w, weighted by
// beta_e (2m+1) h_e^(m-1) / ((2K-1) m! sigma |e|); max over fields.  Then the
// exact OE step: mode (a, b) decays by exp(-tau sum_{m <= min(a+b, K)} delta^m).
// On a face normal to direction n the multi-index is (normal order an,
// tangential order m - an); K's trace sits at normal coordinate s = +-1, the
// overlapping cell's at its centre line (normal coordinate 0).
template <int SYS, int BC, int K, int B, int FORM>
__global__ void __launch_bounds__(NTK, Modes2<K, B>::M > 10 ? 2 : (K > 2 ? 3 : 4))
    k_oe2k(Geo g, OeK oec, const double* __restrict__ uh, double* __restrict__ res, const double* __restrict__ dt,
           const double* __restrict__ sigma, int* __restrict__ status) {
  using MD = Modes2<K, B>;
  constexpr int F = Fields2<SYS>::F, M = MD::M;
  const unsigned full = 0xffffffffu;
  const int mesh = blockIdx.x & 1;
  __shared__ double isg[F];  // 1/sigma of this mesh's fields, once per block
  oe_inv_sigma<F>(sigma, mesh, isg);
  const int lane = threadIdx.x & 31, q = lane >> 3, cl = lane & 7;
  const int sx = q & 1, sy = q >> 1;
  const int tile = blockIdx.x >> 1, tx = (g.nxs + 7) / 8;
  const int i0 = (tile % tx) * 8, j = (tile / tx) * (NTK / 32) + (threadIdx.x >> 5);
  const bool active = i0 + cl < cells_x(g, mesh) && j < cells_y(g, mesh);
  const int ic = active ? i0 + cl : 0, jc = active ? j : 0;
  const long long P = g.plane;
  const int off = mesh == 0 ? -1 : 0;
  bool mx = false, my = false;  // the overlapping cell is a mirror image across a wall
  const int oi = BC == BC_GENERAL ? side_index(g, 0, 1 - mesh, unwrapped(g, 0, mesh, ic) + sx + off, mx)
                                  : wrap_index<BC>(ic + sx + off, g.nx);
  const int oj = BC == BC_GENERAL ? side_index(g, 1, 1 - mesh, unwrapped(g, 1, mesh, jc) + sy + off, my)
                                  : wrap_index<BC>(jc + sy + off, g.ny);
  const double* us = uh + (long long)mesh * F * M * P + (long long)jc * g.nxs + ic;
  const double* uo = uh + (long long)(1 - mesh) * F * M * P + (long long)oj * g.nxs + oi;
  const int fq = F == 4 ? q : 0;  // the field this lane finishes

  fx T[2][K + 1];
  int ev[K + 1];  // the exponents of T's orders
#pragma unroll
  for (int m = 0; m <= K; ++m) ev[m] = 0;
#pragma unroll 1
  for (int f = 0; f < F; ++f) {
    const bool neg = BC == BC_GENERAL && SYS == SYS_EULER && ((mx && f == 1) || (my && f == 2));
    if constexpr (FORM == OEK_DELTA) {
      double S[2 * (K + 1)];
      oe_quarter_fp64<K, B>(us + (long long)(f * M) * P, uo + (long long)(f * M) * P, P,
                            (unsigned)(sx | sy << 1 | (int)mx << 2 | (int)my << 3 | (int)neg << 4), oe_unit(isg[f]), g.i2x,
                            g.i2y, S);
#pragma unroll
      for (int n = 0; n < 2; ++n)
#pragma unroll
        for (int m = 0; m <= K; ++m) {
          double t = S[n * (K + 1) + m] * (1.0 / (oek_rule_unit(K + 1) * (1 << m)));
          t += __shfl_xor_sync(full, t, 8);
          t += __shfl_xor_sync(full, t, 16);
          if (f == fq) T[n][m] = __double_as_longlong(t);
        }
    } else if constexpr (FORM == OEK_OBLONG) {
      fx s[2][K + 1];
      int E[K + 1];
      oek_oblong<K, B, LD_NC>(g, us + (long long)(f * M) * P, uo + (long long)(f * M) * P, sx, sy, mx, my, neg, s, E);
#pragma unroll
      for (int m = 0; m <= K; ++m) {
#pragma unroll
        for (int n = 0; n < 2; ++n) {
          fx t = s[n][m];
          t += shfl_xor_fx(t, 8);
          t += shfl_xor_fx(t, 16);
          if (f == fq) T[n][m] = t;
        }
        if (f == fq) ev[m] = E[m];
      }
    } else {
      double k[M], o[M];
#pragma unroll
      for (int m = 0; m < M; ++m) {
        k[m] = __ldg(us + (long long)(f * M + m) * P);
        o[m] = __ldg(uo + (long long)(f * M + m) * P);
      }
      if (neg) o[0] = -o[0];
      o[0] -= k[0];  // the means' difference; K's own mean counts as 0
      unsigned mag = fx_mag(o[0]);
#pragma unroll
      for (int m = 1; m < M; ++m) mag = max(mag, max(fx_mag(k[m]), fx_mag(o[m])));
      int ex = fx_exp(mag);
      ex = max(ex, __shfl_xor_sync(full, ex, 8));
      ex = max(ex, __shfl_xor_sync(full, ex, 16));
      fx kc[M], oc[M];
      kc[0] = 0;
      oc[0] = to_fx<OEK_FX>(o[0], ex);
#pragma unroll
      for (int m = 1; m < M; ++m) {
        const unsigned fk = (MD::a(m) & 1 ? (unsigned)sx : 0u) ^ (MD::b(m) & 1 ? (unsigned)sy : 0u);
        const unsigned fo = fk ^ (MD::a(m) & 1 ? (unsigned)mx : 0u) ^ (MD::b(m) & 1 ? (unsigned)my : 0u) ^ (unsigned)neg;
        kc[m] = to_fx<OEK_FX>(k[m], ex, fk << 31);
        oc[m] = to_fx<OEK_FX>(o[m], ex, fo << 31);
      }
      fx s[2][K + 1];
      oek_half_face<K, B, 0>(kc, oc, s[0]);
      oek_half_face<K, B, 1>(kc, oc, s[1]);
#pragma unroll
      for (int n = 0; n < 2; ++n)
#pragma unroll
        for (int m = 0; m <= K; ++m) {
          fx t = s[n][m];
          t += shfl_xor_fx(t, 8);
          t += shfl_xor_fx(t, 16);
          if (f == fq) T[n][m] = t;
        }
#pragma unroll
      for (int m = 0; m <= K; ++m)
        if (f == fq) ev[m] = ex;
    }
  }

  // wave speeds at the cell average, delta^m of field fq, the maximum over the fields
  double bx = 0.0, by = 0.0;
  if (SYS == SYS_EULER) {
    const bool ok = euler2_wave(g.gamma, __ldg(us), __ldg(us + (long long)M * P), __ldg(us + (long long)(2 * M) * P),
                                __ldg(us + (long long)(3 * M) * P), bx, by);
    if (!ok && active) atomicOr(status, ST_NONPHYSICAL);
  } else if (SYS == SYS_BURGERS) {
    bx = by = fabs(__ldg(us));
  } else {
    bx = fabs(g.adv_x);
    by = fabs(g.adv_y);
  }
  double d[K + 1];
#pragma unroll
  for (int m = 0; m <= K; ++m) {
    // the sums' unit: 2^(ev - 1023 - OEK_FX)
    const double pw = FORM == OEK_DELTA ? 1.0 / oe_unit(isg[fq]) : __hiloint2double((ev[m] - OEK_FX) << 20, 0);
    const double w = ev[0] >= FX_EXNAN ? __longlong_as_double(0x7ff8000000000000LL) : isg[fq] * pw;
    double tx = FORM == OEK_DELTA ? __longlong_as_double(T[0][m]) : __ll2double_rn(T[0][m]);
    double ty = FORM == OEK_DELTA ? __longlong_as_double(T[1][m]) : __ll2double_rn(T[1][m]);
    if (FORM == OEK_OBLONG && g.hx < g.hy) {  // read transposed
      const double t = tx;
      tx = ty;
      ty = t;
    }
    long long key = oe_key(fma(bx * oec.c[0][m], tx, (by * oec.c[1][m]) * ty) * w);
    if (F == 4) {
      key = max(key, shfl_xor_fx(key, 8));
      key = max(key, shfl_xor_fx(key, 16));
    }
    d[m] = __longlong_as_double(key);
  }
  if (FORM == OEK_DELTA) {
    double* dp = res + (((long long)mesh * g.nys + j) * g.nxs + ic) * (K + 1);
#pragma unroll
    for (int m = 0; m <= K; ++m)
      if (active && q == 0) dp[m] = d[m];
  } else {
    const double tau = dt[0];
    double rate = d[0] + d[1];  // lane q: the decay of degree min(q + 1, K)
#pragma unroll
    for (int m = 2; m <= K; ++m)
      if (q + 1 >= m) rate += d[m];
    const double mine = exp(-tau * rate);
    double e[K + 1];
    e[0] = 1.0;
#pragma unroll
    for (int m = 1; m <= K; ++m) e[m] = __shfl_sync(full, mine, 8 * (m - 1) + cl);
    if (active) {
      double* os = res + (long long)mesh * F * M * P + (long long)j * g.nxs + ic + (long long)(fq * M) * P;
#pragma unroll
      for (int m = 0; m < M; ++m) {
        if (F != 4 && (m & 3) != q) continue;  // one field: its modes over the 4 lanes
        constexpr int KK = K;
        const int deg = MD::a(m) + MD::b(m) < KK ? MD::a(m) + MD::b(m) : KK;
        const double v = __ldg(us + (long long)(fq * M + m) * P);
        os[(long long)m * P] = deg == 0 ? v : v * e[deg];
      }
    }
  }
}

template <int FORM>
static cudaError_t oe2k(int sys, int bc, int k, int basis, const Geo& g, const double* uh, double* res,
                        const double* dt, const double* sigma, int* status, cudaStream_t st) {
  by_sys_bc_k_b(sys, bc, k, basis, [&](auto S, auto Bc, auto Kc, auto Bs) {
    constexpr int S_ = decltype(S)::value, B_ = decltype(Bc)::value, K_ = decltype(Kc)::value;
    constexpr int Q_ = decltype(Bs)::value;
    OeK oec;  // (2m+1) h^(m-1) / ((2K-1) m!) / 4 x (2/min(hx, hy))^m x the integer sums' unit
    double i2 = oek_rule_unit(K_ + 1) * 0.25, hx = g.i1x, hy = g.i1y;
    for (int m = 0; m <= K_; ++m) {
      const double c = i2 * (2 * m + 1) / ((2 * K_ - 1) * fact(m));
      oec.c[0][m] = c * hx;
      oec.c[1][m] = c * hy;
      hx *= g.hx;
      hy *= g.hy;
      i2 *= 2.0 * (g.i2x > g.i2y ? g.i2x : g.i2y);
    }
    k_oe2k<S_, B_, K_, Q_, FORM><<<grid2k(g, NTK / 32), NTK, 0, st>>>(g, oec, uh, res, dt, sigma, status);
  });
  return cudaGetLastError();
}

}  // namespace oecdg
