// oecdg_2d.cu -- 2D Q^2 kernels of the OECDG forward step (arXiv:2503.12473):
// launch wrappers around the per-cell code of oecdg_2d_body.cuh.
#include <type_traits>

#include "oecdg_2d_body.cuh"
#include "oecdg_kernels.h"
#include "oecdg_persist.cuh"

namespace oecdg {

#ifndef OECDG_OE_MINB
#define OECDG_OE_MINB 4
#endif
// MODE_RHS: out = L(uin) with tau_max = dt[1].
// MODE_STAGE: out = ca un + cb (uin + tau L(uin)) with (tau, tau_max) = dt[0..1],
//   plus per-block partials of the sigma reduction of the output:
//   partials[(mesh * nblk + blk) * F * 3 + f * 3 + {0,1,2}] = (sum of cell
//   averages, max and min of the values at the cell's 3x3 Gauss points).
// A block is a tile of 8 x STY cells (stage_block2d); the two meshes' blocks of
// a tile are adjacent in launch order.
constexpr int STY = 4;
template <int SYS, int BC, int MODE>
__global__ void __launch_bounds__(32 * STY, SYS == SYS_EULER ? 3 : 4) k_stage2d(Geo g, const double* __restrict__ uin,
                                                      const double* __restrict__ un, double* __restrict__ out,
                                                      const double* __restrict__ dt, double ca, double cb,
                                                      double* __restrict__ partials) {
  extern __shared__ double smem[];
  constexpr int F = Fields<SYS>::F;
  const int mesh = blockIdx.x & 1, bx = blockIdx.x >> 1, tx = gridDim.x >> 1;
  const long long nblk = (long long)tx * gridDim.y;
  const long long blk = (long long)blockIdx.y * tx + bx;
  stage_block2d<SYS, BC, MODE, LD_NC, STY>(g, uin, un, out, dt, ca, cb, partials + (mesh * nblk + blk) * F * 3, mesh,
                                           bx * SW_CELLS, blockIdx.y * STY, smem);
}

// Fixed-order reduction of the block partials: avg and sigma per mesh and
// field (Section 2.2): avg = mean of the cell averages over the stored cells,
// sigma = max(max - avg, avg - min) over the cell Gauss points.  grid = (F, 2),
// 256 threads each (block_sigma): the same summation order, bit for bit, as the
// one warp per (mesh, field) of the persistent kernels' sigma phase.
__global__ void k_sigma(const double* __restrict__ partials, long long nblk, int F, SigmaNorm sn,
                        double* __restrict__ sigma, double* __restrict__ avg) {
  block_sigma<LD_NC>(partials, nblk, F, blockIdx.y, blockIdx.x, sn, avg, sigma);
}

// ---------------------------------------------------------------- OE step --

// Damping coefficients delta_K^m (m = 0, 1, 2) of one cell and the exact OE
// step (Eq. (OEstep2D)).  For each field and each half-face e of K (k+1 = 3
// Gauss points): the derivatives d^alpha (u^C - u^D), |alpha| <= 2, from K's own
// interior trace and the overlapping cell (which is smooth across e);
//   int_e |u^C - u^D|,  int_e (D_x^2 + D_y^2)^{1/2},  int_e (D_xx^2 + D_xy^2 + D_yy^2)^{1/2}.
// delta^m = sum_e beta_e (2m+1) h_e^{m-1} / ((2k-1) m! sigma |e|) int_e ..., max
// over fields (Remark on systems); delta = 0 where sigma = 0.  Mode (a,b) then
// decays by exp(-tau sum_{m <= min(a+b, 2)} delta^m), the average is kept.
// Damping coefficients and the exact OE step of every cell (oe_warp2d).
template <int SYS, int BC, int FORM>
__global__ void __launch_bounds__(32 * STY, OECDG_OE_MINB) k_oe2d(Geo g, const double* __restrict__ uh,
                                                                  double* __restrict__ usig,
                                                                  const double* __restrict__ dt,
                                                                  const double* __restrict__ sigma,
                                                                  int* __restrict__ status) {
  __shared__ double isg[Fields<SYS>::F];
  oe_inv_sigma<Fields<SYS>::F>(sigma, blockIdx.x & 1, isg);
  oe_warp2d<SYS, BC, 0, FORM, LD_NC>(g, uh, usig, dt, isg, status, blockIdx.x & 1,
                                                 (blockIdx.x >> 1) * SW_CELLS, blockIdx.y * STY + (threadIdx.x >> 5));
}

// ------------------------------------------------------------- time step --

// Per-block maximum wave speeds over the cell averages of both meshes.
// partial[blk * 2 + {0,1}] = (max |u| + c, max |v| + c) (advection: |a_x|, |a_y|).
template <int SYS>
__global__ void k_wave2d(Geo g, const double* __restrict__ u, double* __restrict__ partial, int* __restrict__ status) {
  constexpr int F = Fields<SYS>::F;
  __shared__ double sh[32];
  const long long n = 2 * g.plane;
  double mx = 0.0, my = 0.0;
  for (long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x; c < n; c += (long long)gridDim.x * blockDim.x) {
    const int mesh = (int)(c / g.plane);
    const long long cell = c - mesh * g.plane;
    const double* us = u + (long long)mesh * F * 9 * g.plane + cell;
    if (SYS == SYS_EULER) {
      double bx, by;
      if (euler2_wave(g.gamma, us[0], us[9 * g.plane], us[18 * g.plane], us[27 * g.plane], bx, by)) {
        mx = fmax(mx, bx);
        my = fmax(my, by);
      } else {
        atomicOr(status, ST_NONPHYSICAL);
      }
    } else {
      mx = fabs(g.adv_x);
      my = fabs(g.adv_y);
    }
  }
  mx = block_reduce_max(mx, sh);
  __syncthreads();
  my = block_reduce_max(my, sh);
  if (threadIdx.x == 0) {
    partial[blockIdx.x * 2] = mx;
    partial[blockIdx.x * 2 + 1] = my;
  }
}

// One block: the maxima of the block partials (exact in any order), then
// finish_dt (tau_max, the clipped tau, the time) by thread 0.
__global__ void k_dt_final(const double* __restrict__ partial, int nblk, double hx, double hy, int dim, double cfl,
                           double T_end, double* __restrict__ dt, double* __restrict__ time) {
  __shared__ double sh[32];
  double bx = 0.0, by = 0.0;
  for (int b = threadIdx.x; b < nblk; b += blockDim.x) {
    bx = fmax(bx, partial[2 * b]);
    by = fmax(by, partial[2 * b + 1]);
  }
  bx = block_reduce_max(bx, sh);
  __syncthreads();
  by = block_reduce_max(by, sh);
  if (threadIdx.x == 0) finish_dt(bx, by, hx, hy, dim, cfl, T_end, dt, time);
}

__global__ void k_set2(double* __restrict__ p, double a, double b) {
  if (threadIdx.x == 0 && blockIdx.x == 0) {
    p[0] = a;
    p[1] = b;
  }
}

// ------------------------------------------------------ initial projection --

// Composite-Gauss sampling points, layout [mesh][j][i][sy][sx][qy][qx] (x, y).
__global__ void k_points2d(Geo g, double ax, double ay, double* __restrict__ xy) {
  const long long n = 2 * g.plane * 36;
  for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < n; t += (long long)gridDim.x * blockDim.x) {
    const int r = (int)(t % 36);
    const long long c = t / 36;
    const int mesh = (int)(c / g.plane);
    const long long cell = c - mesh * g.plane;
    const int j = (int)(cell / g.nx), i = (int)(cell - (long long)j * g.nx);
    const int qx = r % 3, qy = (r / 3) % 3, sx = (r / 9) % 2, sy = r / 18;
    const double xc = ax + (i + 0.5 + 0.5 * mesh) * g.hx, yc = ay + (j + 0.5 + 0.5 * mesh) * g.hy;
    xy[2 * t] = xc + 0.5 * g.hx * xs_self(sx, qx);
    xy[2 * t + 1] = yc + 0.5 * g.hy * xs_self(sy, qy);
  }
}

// u_ab = (2a+1)(2b+1)/4 * sum over the 4 sub-cells and their 3x3 points of
// (w_qx/2)(w_qy/2) u0 P_a(xi) P_b(eta).
template <int F>
__global__ void k_project2d(Geo g, const double* __restrict__ vals, double* __restrict__ u) {
  const long long n = 2 * g.plane;
  for (long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x; c < n; c += (long long)gridDim.x * blockDim.x) {
    const int mesh = (int)(c / g.plane);
    const long long cell = c - mesh * g.plane;
    double acc[F][9];
#pragma unroll
    for (int f = 0; f < F; ++f)
#pragma unroll
      for (int m = 0; m < 9; ++m) acc[f][m] = 0.0;
    const double* v = vals + c * 36 * F;
#pragma unroll
    for (int r = 0; r < 36; ++r) {
      const int qx = r % 3, qy = (r / 3) % 3, sx = (r / 9) % 2, sy = r / 18;
      const double xi = xs_self(sx, qx), eta = xs_self(sy, qy);
      const double w = 0.25 * gwt(qx) * gwt(qy);
#pragma unroll
      for (int f = 0; f < F; ++f) {
        const double x = w * v[r * F + f];
#pragma unroll
        for (int m = 0; m < 9; ++m) acc[f][m] = fma(x, lp(m % 3, xi) * lp(m / 3, eta), acc[f][m]);
      }
    }
    double* o = u + (long long)mesh * F * 9 * g.plane + cell;
#pragma unroll
    for (int f = 0; f < F; ++f)
#pragma unroll
      for (int m = 0; m < 9; ++m) o[(f * 9 + m) * g.plane] = acc[f][m] * ((2 * (m % 3) + 1) * (2 * (m / 3) + 1) / 4.0);
  }
}

// ----------------------------------------------------------------- launch --

// The two meshes' blocks of a tile are adjacent in launch order (mesh =
// blockIdx.x & 1), so the cells a block reads from the other mesh were just
// read by its partner block and are still in L2: each state is read from DRAM
// about once per launch instead of once per mesh.
static inline dim3 stage_grid(const Geo& g) {
  return dim3(2 * ((g.nxs + SW_CELLS - 1) / SW_CELLS), (g.nys + STY - 1) / STY, 1);
}

long long partial_blocks_2d(const Geo& g) {
  return (long long)((g.nxs + SW_CELLS - 1) / SW_CELLS) * ((g.nys + STY - 1) / STY);
}

template <int SYS, int BC, int MODE>
static cudaError_t stage2d_m(const Geo& g, const double* uin, const double* un, double* out, const double* dt,
                             double ca, double cb, double* partials, cudaStream_t st) {
  constexpr int smem = STY * StageSmem<SYS>::WARP * (int)sizeof(double);
  auto kern = k_stage2d<SYS, BC, MODE>;
  if (smem > 0) {
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
  }
  kern<<<stage_grid(g), 32 * STY, smem, st>>>(g, uin, un, out, dt, ca, cb, partials);
  return cudaGetLastError();
}

template <int SYS, int BC>
static cudaError_t stage2d_t(const Geo& g, int mode, const double* uin, const double* un, double* out, const double* dt,
                             double ca, double cb, double* partials, cudaStream_t st) {
  return mode == MODE_RHS ? stage2d_m<SYS, BC, MODE_RHS>(g, uin, un, out, dt, ca, cb, partials, st)
                          : stage2d_m<SYS, BC, MODE_STAGE>(g, uin, un, out, dt, ca, cb, partials, st);
}

cudaError_t launch_stage2d(int sys, int bc, const Geo& g, int rhs_only, const double* uin, const double* un,
                           double* out, const double* dt, double ca, double cb, double* partials, cudaStream_t st) {
  const int mode = rhs_only ? MODE_RHS : MODE_STAGE;
  auto go = [&](auto S) {
    constexpr int SYS = decltype(S)::value;
    if (bc == BC_PERIODIC) return stage2d_t<SYS, BC_PERIODIC>(g, mode, uin, un, out, dt, ca, cb, partials, st);
    if (bc == BC_TRANSMISSIVE) return stage2d_t<SYS, BC_TRANSMISSIVE>(g, mode, uin, un, out, dt, ca, cb, partials, st);
    return stage2d_t<SYS, BC_GENERAL>(g, mode, uin, un, out, dt, ca, cb, partials, st);
  };
  if (sys == SYS_EULER) return go(std::integral_constant<int, SYS_EULER>{});
  return go(std::integral_constant<int, SYS_ADV>{});
}

cudaError_t launch_sigma(const double* partials, long long nblk, int F, const SigmaNorm& sn, double* sigma,
                         double* avg, cudaStream_t st) {
  k_sigma<<<dim3(F, 2), 256, 0, st>>>(partials, nblk, F, sn, sigma, avg);
  return cudaGetLastError();
}

template <int SYS, int BC>
static cudaError_t oe2d_t(const Geo& g, const double* uh, double* usig, const double* dt, const double* sigma,
                          int* status, cudaStream_t st) {
  const int form = oe_form(g);
  if (form == OE_SQUARE) k_oe2d<SYS, BC, OE_SQUARE><<<stage_grid(g), 32 * STY, 0, st>>>(g, uh, usig, dt, sigma, status);
  else if (form == OE_MILD) k_oe2d<SYS, BC, OE_MILD><<<stage_grid(g), 32 * STY, 0, st>>>(g, uh, usig, dt, sigma, status);
  else k_oe2d<SYS, BC, OE_OBLONG><<<stage_grid(g), 32 * STY, 0, st>>>(g, uh, usig, dt, sigma, status);
  return cudaGetLastError();
}

cudaError_t launch_oe2d(int sys, int bc, const Geo& g, const double* uh, double* usig, const double* dt,
                        const double* sigma, int* status, cudaStream_t st) {
  auto go = [&](auto S) {
    constexpr int SYS = decltype(S)::value;
    if (bc == BC_PERIODIC) return oe2d_t<SYS, BC_PERIODIC>(g, uh, usig, dt, sigma, status, st);
    if (bc == BC_TRANSMISSIVE) return oe2d_t<SYS, BC_TRANSMISSIVE>(g, uh, usig, dt, sigma, status, st);
    return oe2d_t<SYS, BC_GENERAL>(g, uh, usig, dt, sigma, status, st);
  };
  if (sys == SYS_EULER) return go(std::integral_constant<int, SYS_EULER>{});
  return go(std::integral_constant<int, SYS_ADV>{});
}

int wave_blocks_2d(const Geo& g) {
  const long long n = 2 * g.plane;
  long long b = (n + 255) / 256;
  return (int)(b < 1184 ? b : 1184);
}

cudaError_t launch_dt2d(int sys, const Geo& g, const double* u, double* partial, int nblk, double T_end,
                        double* dt, double* time, int* status, cudaStream_t st) {
  if (sys == SYS_EULER) k_wave2d<SYS_EULER><<<nblk, 256, 0, st>>>(g, u, partial, status);
  else k_wave2d<SYS_ADV><<<nblk, 256, 0, st>>>(g, u, partial, status);
  k_dt_final<<<1, 256, 0, st>>>(partial, nblk, g.hx, g.hy, 2, g.cfl, T_end, dt, time);
  return cudaGetLastError();
}

cudaError_t launch_dt_final(const double* partial, int nblk, double hx, double hy, int dim, double cfl, double T_end,
                            double* dt, double* time, cudaStream_t st) {
  k_dt_final<<<1, 256, 0, st>>>(partial, nblk, hx, hy, dim, cfl, T_end, dt, time);
  return cudaGetLastError();
}

cudaError_t launch_set2(double* p, double a, double b, cudaStream_t st) {
  k_set2<<<1, 32, 0, st>>>(p, a, b);
  return cudaGetLastError();
}

cudaError_t launch_points2d(const Geo& g, double ax, double ay, double* xy, cudaStream_t st) {
  k_points2d<<<1184, 256, 0, st>>>(g, ax, ay, xy);
  return cudaGetLastError();
}

cudaError_t launch_project2d(int sys, const Geo& g, const double* vals, double* u, cudaStream_t st) {
  if (sys == SYS_EULER) k_project2d<4><<<1184, 128, 0, st>>>(g, vals, u);
  else k_project2d<1><<<1184, 128, 0, st>>>(g, vals, u);
  return cudaGetLastError();
}

}  // namespace oecdg
