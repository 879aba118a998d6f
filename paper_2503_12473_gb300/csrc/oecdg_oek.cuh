// oecdg_oek.cuh -- the OE step's sums over a quarter's half-faces in fixed point, for
// the 2D spaces Q^k and P^k (arXiv:2503.12473, Section 2.2).
#pragma once

#include "oecdg_fix.cuh"
#include "oecdg_modes.cuh"
#include "oecdg_persist.cuh"

namespace oecdg {

// ------------------------------------------------- rules, fixed point --

// the nodes and weights of the N-point rules times 2^64, all below 2^63
constexpr fx FXN2_T_2 = 0x49e69d1640cc7135LL;    // (1/sqrt 3) / 2
constexpr fx FXN3_TT_2 = 0x4ccccccccccccccdLL;   // (3/5) / 2
__host__ __device__ constexpr fx fxn4_t_2(int k) { return k == 0 ? 0x2b847fb3ba7bf845LL : 0x6e39b6f3d8e61419LL; }     // inner, outer node / 2
__host__ __device__ constexpr fx fxn4_tt_2(int k) { return k == 0 ? 0x0ecb8ef4a3638ce9LL : 0x5eeb4c791377e0ceLL; }  // their squares / 2
constexpr fx FXN4_W_IN_2 = 0x53797e10309329b9LL, FXN4_W_OUT = 0x590d03df9ed9ac8dLL;

// A + B t + C t^2 + D t^3 (p[0..3]) at the N-point rule's nodes, in mirrored pairs
template <int N>
__device__ __forceinline__ void oek_nodes(const fx (&p)[4], fx (&v)[N]) {
  if constexpr (N == 2) {
    const fx o = fx_mul(p[1] << 1, FXN2_T_2);
    v[0] = p[0] - o;
    v[1] = p[0] + o;
  } else if constexpr (N == 3) {
    const fx e = p[0] + fx_mul(p[2] << 1, FXN3_TT_2), o = fx_mul(p[1] << 1, FXK_HALFG);
    v[0] = e - o;
    v[1] = p[0];
    v[2] = e + o;
  } else {
#pragma unroll
    for (int k = 0; k < 2; ++k) {  // v[0], v[1]: inner nodes, v[2], v[3]: outer ones
      const fx e = p[0] + fx_mul(p[2] << 1, fxn4_tt_2(k));
      const fx o = fx_mul((p[1] + fx_mul(p[3] << 1, fxn4_tt_2(k))) << 1, fxn4_t_2(k));
      v[2 * k] = e - o;
      v[2 * k + 1] = e + o;
    }
  }
}
// 1/8 of the rule's sum (N = 3: of 9/4 of it)
template <int N>
__device__ __forceinline__ fx oek_rule(const fx (&v)[N]) {
  if constexpr (N == 2) {
    return (v[0] + v[1] + 4) >> 3;
  } else if constexpr (N == 3) {
    const fx h = (v[0] + v[2]) >> 1;
    return (h + ((h + 2) >> 2) + v[1] + 2) >> 2;
  } else {
    return ((fx_mul(v[0] + v[1], FXN4_W_IN_2) << 1) + fx_mul(v[2] + v[3], FXN4_W_OUT) + 4) >> 3;
  }
}
constexpr double oek_rule_unit(int N) { return N == 3 ? 32.0 / 9.0 : 8.0; }

// ------------------------------------------------------------------ sums --
//
// The damping coefficients on the integer pipes, as in the tiled Q^2 kernel
// (oecdg_2d_body.cuh, where the layout, the scaling and the norm are described):
// a warp owns 8 cells and their 4 quarters, lane = 8 q + c.  Order m is held
// 2^-m smaller, so that one scale serves all: with coefficients below 2^56 every
// derivative stays below 32 2^56 = 2^61 (Q^3, second mixed derivative: K
// (1+3+6)^2, the overlapping cell 5/2 (1+3+6), over 4) and the norms of an order
// below 45 2^56, twice which is a rule's largest sum.
constexpr int OEK_FX = 55;

// P_a^(d) at -1 and 2 P_a^(d) at 0
__host__ __device__ constexpr int oek_low(int a, int d) { return (int)lpd(a, d, -1.0); }
__host__ __device__ constexpr int oek_mid2(int a, int d) { return (int)(2.0 * lpd(a, d, 0.0)); }

// index of the mode of normal degree an and tangential degree at (DIR: the normal), -1: none
template <int K, int B, int DIR>
__host__ __device__ constexpr int oek_mode(int an, int at) {
  const int a = DIR == 0 ? an : at, b = DIR == 0 ? at : an;
  return B == BASIS_Q ? b * (K + 1) + a : (a + b > K ? -1 : (a + b) * (a + b + 1) / 2 + b);
}

// The difference's derivative of normal order an and tangential order at along a
// half-face (normal direction DIR) as a polynomial in t, times 2^-(an + at).  kc, oc:
// K's and the overlapping cell's coefficients in mirrored coordinates (K's face at -1,
// its half at zeta = (t - 1)/2; the overlapping cell's centre line, zeta' = (t + 1)/2),
// of which those of normal degree an and tangential degree at or more are read.
template <int K, int B, int DIR>
__device__ __forceinline__ void oek_poly(int an, int at, const fx (&kc)[Modes2<K, B>::M],
                                         const fx (&oc)[Modes2<K, B>::M], fx (&p)[4]) {
  fx e[4] = {0, 0, 0, 0}, s[4] = {0, 0, 0, 0};
#pragma unroll
  for (int b = 0; b <= K; ++b) {
    if (b < at) continue;
    fx k = 0, o2 = 0;
#pragma unroll
    for (int a = 0; a <= K; ++a) {
      const int m = oek_mode<K, B, DIR>(a, b);
      if (a >= an && m >= 0) {
        k += oek_low(a, an) * kc[m];
        o2 += oek_mid2(a, an) * oc[m];
      }
    }
    fx o = o2 >> 1;
    if (an > 0) {
      k = (k + ((1 << an) >> 1)) >> an;
      o = (o + ((1 << an) >> 1)) >> an;
    }
    e[b] = k - o;
    s[b] = k + o;
  }
  p[1] = p[2] = p[3] = 0;
  if (at == 0) {
    p[0] = e[0] - (s[1] >> 1) - (e[2] >> 3) + ((7 * s[3]) >> 4);
    p[1] = (e[1] >> 1) - ((3 * s[2]) >> 2) + ((3 * e[3]) >> 4);
    p[2] = ((3 * e[2]) >> 3) - ((15 * s[3]) >> 4);
    p[3] = (5 * e[3]) >> 4;
  } else if (at == 1) {
    p[0] = (e[1] - s[2] - (s[2] >> 1) + ((3 * e[3]) >> 3)) >> 1;
    p[1] = (3 * e[2] - ((15 * s[3]) >> 1)) >> 2;
    p[2] = (15 * e[3]) >> 4;
  } else if (at == 2) {
    p[0] = (3 * e[2] - ((15 * s[3]) >> 1)) >> 2;
    p[1] = (15 * e[3]) >> 3;
  } else {
    p[0] = (15 * e[3]) >> 3;
  }
}

// The rule's sum (oek_rule) of the norm of order m from its m + 1 derivatives at the points
template <int K>
__device__ __forceinline__ fx oek_norm_sum(int m, const fx (&v)[K + 1][K + 1]) {
  constexpr int N = K + 1;
  fx r[N];
#pragma unroll
  for (int q = 0; q < N; ++q) {
    if (m == 0) r[q] = fx_abs(v[0][q]);
    else if (m == 1) r[q] = fx_norm(v[0][q], v[1 <= K ? 1 : 0][q]);
    else if (m == 2) r[q] = fx_norm(v[0][q], v[1][q], v[2 <= K ? 2 : 0][q]);
    else r[q] = fx_norm(v[0][q], v[1][q], v[2 <= K ? 2 : 0][q], v[3 <= K ? 3 : 0][q]);
  }
  return oek_rule<N>(r);
}

// One half-face of a square cell: S[m] = the rule's sum of the order-m norm.
template <int K, int B, int DIR>
__device__ __forceinline__ void oek_half_face(const fx (&kc)[Modes2<K, B>::M], const fx (&oc)[Modes2<K, B>::M],
                                              fx (&S)[K + 1]) {
#pragma unroll
  for (int m = 0; m <= K; ++m) {
    fx v[K + 1][K + 1];
#pragma unroll
    for (int an = 0; an <= m; ++an) {
      fx p[4];
      oek_poly<K, B, DIR>(an, m - an, kc, oc, p);
      oek_nodes<K + 1>(p, v[an]);
    }
    S[m] = oek_norm_sum<K>(m, v);
  }
}

// Oblong cells.  A derivative of order al along the longer side counts rho^al, rho =
// h_min / h_max, and delta^m takes the norm of order m times up to rho^(1-m) more than
// the shorter side's faces do: one exponent for all coefficients cut the derivatives
// along the shorter side too early (P^3 at rho = 10^-4: 5e-11 of a damped mode), and rho^m
// in 62 bits those along the longer one.  So
//   - the coefficients of degree j or more along the shorter side have an exponent G[j]
//     of their own, and a derivative of order j along it takes them under that;
//   - each order has its exponent E[m], that of its largest scaled derivative, and the
//     factors rho^al 2^(G[m - al] - E[m]) are taken from normalised mantissas (g.rho).
// In coordinates with the shorter side along y: with hx < hy the modes and the quarter
// are read transposed, and S[0], S[1] are then the half-faces normal to y and x.
// S[d][m]: the rule's sums in units of 2^(E[m] - 1023 - OEK_FX) 2^m / h_min^m.
// Measured, a launch of the OE step against that with one exponent: P^3 256 x 250 0.42 ->
// 0.40 ms, P^2 512 x 500 0.56 -> 0.51 ms, Q^3 256 x 250 0.67 -> 0.77 ms (its 255 registers).
template <int K, int B, int LD>
__device__ __forceinline__ void oek_oblong(const Geo& g, const double* __restrict__ us, const double* __restrict__ uo,
                                           int sx, int sy, int mx, int my, int neg, fx (&S)[2][K + 1],
                                           int (&E)[K + 1]) {
  using MD = Modes2<K, B>;
  constexpr int M = MD::M;
  const unsigned full = 0xffffffffu;
  const long long P = g.plane;
  const bool swap = g.hx < g.hy;
  if (swap) {
    int t = sx;
    sx = sy;
    sy = t;
    t = mx;
    mx = my;
    my = t;
  }
  double k[M], o[M];
  // transposed, Q^k's modes (a, b) lie at a (K+1) + b, P^k's of a total degree in reverse
  const long long da = B == BASIS_P ? 0 : (swap ? (K + 1) * P : P);
  const long long db = B == BASIS_P ? (swap ? -P : P) : (swap ? P : (K + 1) * P);
#pragma unroll
  for (int m = 0; m < M; ++m) {
    const int s = MD::a(m) + MD::b(m);
    const long long row = B == BASIS_Q ? 0 : (s * (s + 1) / 2 + (swap ? s : 0)) * P;
    const long long at = row + MD::a(m) * da + MD::b(m) * db;
    k[m] = ldv<LD>(us + at);
    o[m] = ldv<LD>(uo + at);
  }
  if (neg) o[0] = -o[0];
  o[0] -= k[0];  // the means' difference; K's own mean counts as 0
  int G[K + 1];
  {
    unsigned mag = 0;
#pragma unroll
    for (int j = K; j >= 0; --j) {
#pragma unroll
      for (int m = 0; m < M; ++m)
        if (MD::b(m) == j) mag = max(mag, max(m == 0 ? 0u : fx_mag(k[m]), fx_mag(o[m])));
      G[j] = fx_exp(mag);
      G[j] = max(G[j], __shfl_xor_sync(full, G[j], 8));
      G[j] = max(G[j], __shfl_xor_sync(full, G[j], 16));
    }
  }
  fx kc[K + 1][M], oc[K + 1][M];  // [exponent G[j]]
#pragma unroll
  for (int m = 0; m < M; ++m) {
    const unsigned fk = (MD::a(m) & 1 ? (unsigned)sx : 0u) ^ (MD::b(m) & 1 ? (unsigned)sy : 0u);
    const unsigned fo = fk ^ (MD::a(m) & 1 ? (unsigned)mx : 0u) ^ (MD::b(m) & 1 ? (unsigned)my : 0u) ^
                        (m > 0 ? (unsigned)neg : 0u);
#pragma unroll
    for (int j = K; j >= 0; --j) {
      if (j > MD::b(m)) continue;
      if (j == MD::b(m)) {
        kc[j][m] = m == 0 ? 0 : to_fx<OEK_FX>(k[m], G[j], fk << 31);
        oc[j][m] = to_fx<OEK_FX>(o[m], G[j], fo << 31);
      } else {
        kc[j][m] = fx_shr(kc[j + 1][m], G[j] - G[j + 1]);
        oc[j][m] = fx_shr(oc[j + 1][m], G[j] - G[j + 1]);
      }
    }
  }
#pragma unroll
  for (int m = 0; m <= K; ++m) {
    E[m] = G[m];
#pragma unroll
    for (int al = 1; al <= m; ++al) E[m] = max(E[m], G[m - al] - g.rho_x[al - 1]);
    fx vx[K + 1][K + 1], vy[K + 1][K + 1];  // half-faces normal to x (an = al) and to y (at = al)
#pragma unroll
    for (int al = 0; al <= m; ++al) {
      const int as = m - al;
      fx px[4], py[4];
      oek_poly<K, B, 0>(al, as, kc[as], oc[as], px);
      oek_poly<K, B, 1>(as, al, kc[as], oc[as], py);
      if (al == 0) {
        const int s = E[m] - G[as];
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          px[c] = fx_shr(px[c], s);
          py[c] = fx_shr(py[c], s);
        }
      } else {
        const FxLimbs r(fx_shr(g.rho[al - 1], g.rho_x[al - 1] - G[as] + E[m]));
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          if (c <= (B == BASIS_P ? K - m : K - as)) px[c] = fx_prod(FxLimbs(px[c]), r);
          if (c <= (B == BASIS_P ? K - m : K - al)) py[c] = fx_prod(FxLimbs(py[c]), r);
        }
      }
      oek_nodes<K + 1>(px, vx[al]);
      oek_nodes<K + 1>(py, vy[as]);
    }
    S[0][m] = oek_norm_sum<K>(m, vx);
    S[1][m] = oek_norm_sum<K>(m, vy);
  }
}

}  // namespace oecdg
