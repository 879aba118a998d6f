// oecdg_batch.cu -- many independent 2D Q^2 OECDG problems of uneven mesh
// sizes advanced together (arXiv:2503.12473 applied to a batch of meshes).
//
// Every phase of a step is ONE launch over all instances: the blocks of the
// stage and OE kernels are laid out instance after instance (2 meshes x tiles
// of 8 x R cells each), and a block finds its instance by binary search over
// the instances' first-block offsets.  Reductions (sigma, wave speed) and the
// time step are kept per instance, so each instance evolves exactly as it
// would alone (bitwise, for the same tile height R = 4 as the single-mesh
// kernels).  A step is 11 launches whatever the number of instances, and
// cdg_batch_step can capture the launches of nsteps steps in a CUDA graph.
// The persistent mode runs nsteps steps of every instance in ONE cooperative
// launch (k_bpersist): its blocks loop over the same tiles phase by phase and
// meet at grid-wide barriers with a bounded wait (CDG_ETIMEOUT when a wait
// runs out); it runs the same per-cell code and the same fixed-order
// reductions, so its results equal the per-phase launches' bit for bit.
// The tile height R (2, 4 or 8 rows) and the persistent grid (blocks per SM)
// are picked by cdg_batch_autotune.
#include <cuda_runtime.h>
#include <stdio.h>
#include <stdlib.h>
#include <string.h>

#include "../../include/oecdg.h"
#include "oecdg_2d_body.cuh"
#include "oecdg_kernels.h"
#include "oecdg_persist.cuh"

namespace oecdg {

struct BatchInst {
  Geo g;
  double* u;      // caller's state (u^n, and u^{n+1} after the last stage)
  double* a;      // scratch u_h
  double* b;      // scratch u_sigma
  double* part;   // sigma partials [2][tiles][F][3]
  double* wpart;  // wave-speed partials [WB][2]
  double* dt;     // [tau, tau_max]
  double* time;   // [t, unused]
  double* sigma;  // [2][F]
  double* avg;    // [2][F]
  long long blk0; // first block of this instance
  int tx, ty;     // tiles (8 x R cells) per direction (per mesh)
};

constexpr int WB = 32;  // wave-speed blocks per instance

__device__ __forceinline__ int find_instance(const BatchInst* __restrict__ I, int n, long long blk) {
  int lo = 0, hi = n - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (I[mid].blk0 <= blk) lo = mid;
    else hi = mid - 1;
  }
  return lo;
}

// stage block `blk` of the batch: its instance, mesh and tile, then the tile
template <int SYS, int BC, int R, int LD>
__device__ __forceinline__ void bstage_tile(const BatchInst* __restrict__ I, int n, long long blk, int l, double ca,
                                            double cb, double* smem) {
  constexpr int F = Fields<SYS>::F;
  const BatchInst& in = I[find_instance(I, n, blk)];
  const int tiles = in.tx * in.ty;
  const int local = (int)(blk - in.blk0);
  const int mesh = local & 1, t = local >> 1;  // the two meshes' blocks of a tile side by side
  stage_block2d<SYS, BC, MODE_STAGE, LD, R>(in.g, l == 0 ? in.u : in.b, in.u, in.a, in.dt, ca, cb,
                                            in.part + ((long long)mesh * tiles + t) * F * 3, mesh,
                                            (t % in.tx) * SW_CELLS, (t / in.tx) * R, smem);
}

template <int SYS, int BC, int R>
__global__ void __launch_bounds__(32 * R, R == 8 ? 1 : 12 / R) k_bstage(const BatchInst* __restrict__ I, int n, int l, double ca,
                                                   double cb) {
  extern __shared__ double smem[];
  bstage_tile<SYS, BC, R, LD_NC>(I, n, blockIdx.x, l, ca, cb, smem);
}

// OE block `blk` of the batch: the damping coefficients and the OE step of its tile.
// SQUARE: every instance has square cells (with the other forms beside it the kernel of
// 256 such meshes spills registers: a step of 11 launches 446.0 ms, against 443.6)
template <int SYS, int BC, int R, int LD, bool SQUARE>
__device__ __forceinline__ void boe_tile(const BatchInst* __restrict__ I, int n, long long blk, int last,
                                         double* isg, int* __restrict__ status) {
  const BatchInst& in = I[find_instance(I, n, blk)];
  const int local = (int)(blk - in.blk0);
  const int mesh = local & 1, t = local >> 1;
  const int i0 = (t % in.tx) * SW_CELLS, j = (t / in.tx) * R + (threadIdx.x >> 5);
  double* out = last ? in.u : in.b;
  oe_inv_sigma<Fields<SYS>::F>(in.sigma, mesh, isg);
  const int form = oe_form(in.g);  // as the single-mesh launch
  if (SQUARE || form == OE_SQUARE) oe_warp2d<SYS, BC, 0, OE_SQUARE, LD>(in.g, in.a, out, in.dt, isg, status, mesh, i0, j);
  else if (form == OE_MILD) oe_warp2d<SYS, BC, 0, OE_MILD, LD>(in.g, in.a, out, in.dt, isg, status, mesh, i0, j);
  else oe_warp2d<SYS, BC, 0, OE_OBLONG, LD>(in.g, in.a, out, in.dt, isg, status, mesh, i0, j);
}

template <int SYS, int BC, int R, bool SQUARE>
__global__ void __launch_bounds__(32 * R, 16 / R) k_boe(const BatchInst* __restrict__ I, int n, int last,
                                                        int* __restrict__ status) {
  __shared__ double isg[Fields<SYS>::F];
  boe_tile<SYS, BC, R, LD_NC, SQUARE>(I, n, blockIdx.x, last, isg, status);
}

// avg and sigma per instance, mesh and field: grid (F, 2, n), one warp each,
// the fixed-order reduction shared with every other path
__global__ void k_bsigma(const BatchInst* __restrict__ I, int F) {
  const BatchInst& in = I[blockIdx.z];
  warp_sigma<LD_NC>(in.part, (long long)in.tx * in.ty, F, blockIdx.y, blockIdx.x, plain_norm(in.g.plane), in.avg,
                    in.sigma);
}

// per-instance maximum wave speeds over both meshes' cell averages: chunk ch
// of WB takes cells ch * blockDim.x + threadIdx.x, strided by WB * blockDim.x
template <int SYS, int LD>
__device__ __forceinline__ void bwave_chunk(const BatchInst& in, int ch, int* __restrict__ status) {
  constexpr int F = Fields<SYS>::F;
  const Geo& g = in.g;
  __shared__ double sh[32];
  const long long nc = 2 * g.plane;
  double mx = 0.0, my = 0.0;
  for (long long c = (long long)ch * blockDim.x + threadIdx.x; c < nc; c += (long long)WB * blockDim.x) {
    const int mesh = (int)(c / g.plane);
    const long long cell = c - mesh * g.plane;
    const double* us = in.u + (long long)mesh * F * 9 * g.plane + cell;
    if (SYS == SYS_EULER) {
      double bx, by;
      if (euler2_wave(g.gamma, ldv<LD>(us), ldv<LD>(us + 9 * g.plane), ldv<LD>(us + 18 * g.plane),
                      ldv<LD>(us + 27 * g.plane), bx, by)) {
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
    in.wpart[ch * 2] = mx;
    in.wpart[ch * 2 + 1] = my;
  }
  __syncthreads();  // sh is reused by the next chunk
}

// grid (WB, n)
template <int SYS>
__global__ void k_bwave(const BatchInst* __restrict__ I, int* __restrict__ status) {
  bwave_chunk<SYS, LD_NC>(I[blockIdx.y], blockIdx.x, status);
}

// tau_max of one instance from its WB wave partials (no end time): the time
// step of Section 4, as finish_dt without clipping
template <int LD>
__device__ __forceinline__ void bdt_instance(const BatchInst& in) {
  double bx = 0.0, by = 0.0;
  for (int b = 0; b < WB; ++b) {
    bx = fmax(bx, ldv<LD>(in.wpart + 2 * b));
    by = fmax(by, ldv<LD>(in.wpart + 2 * b + 1));
  }
  const double rate = bx / in.g.hx + by / in.g.hy;
  const double tm = rate > 0.0 ? in.g.cfl / rate : 0.0;
  in.dt[0] = tm;
  in.dt[1] = tm > 0.0 ? tm : 1.0;
  in.time[0] += tm;  // written only here, by the thread that owns instance q in every step
}

// tau_max = C_CFL / (beta_x/h_x + beta_y/h_y) per instance (no end time)
__global__ void k_bdt(const BatchInst* __restrict__ I, int n) {
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q < n) bdt_instance<LD_NC>(I[q]);
}

// ------------------------------------------------------- persistent step --

__constant__ double BSSP3_CA[3] = {0.0, 0.75, 1.0 / 3.0};

struct BPersistArgs {
  const BatchInst* I;
  int n;
  long long ntiles;             // tiles of all instances, both meshes (= the per-phase grids)
  int nsteps;
  unsigned long long* bar;      // barrier arrival counter, zeroed before the launch
  unsigned long long expected;  // arrivals per barrier: gridDim.x (+ withheld ones in a test)
  unsigned long long limit_ns;  // bounded wait of every barrier
  int* status;
  int stages;                   // 3 (the SSP-RK3 step); 1 when the autotuner times a first stage only
};

// nsteps SSP-RK3 steps of every instance in one cooperative launch.  Phases
// (each ends at a grid barrier): wave-speed chunks (instance x WB) -> tau per
// instance -> 3 x [stage tiles -> sigma (one warp per instance, mesh and
// field) -> OE tiles].  Block b takes the items b, b + gridDim.x, ... of every
// phase; data written in one phase are read in a later one with plain loads
// (LD_CA), ordered by the barriers' fences.  A barrier that runs out of time
// sets ST_TIMEOUT and every block returns.
template <int SYS, int BC, int R>
__global__ void __launch_bounds__(32 * R) k_bpersist(BPersistArgs a) {
  extern __shared__ double smem[];
  constexpr int F = Fields<SYS>::F;
  __shared__ double isg[F];  // 1/sigma of the OE phase's current tile (its instance and mesh)
  const long long nwave = (long long)a.n * WB;
  for (int s = 0; s < a.nsteps; ++s) {
    for (long long it = blockIdx.x; it < nwave; it += gridDim.x)
      bwave_chunk<SYS, LD_CA>(a.I[it / WB], (int)(it % WB), a.status);
    if (!grid_sync(a.bar, a.expected, a.status, a.limit_ns)) return;
    for (long long q = (long long)blockIdx.x * blockDim.x + threadIdx.x; q < a.n;
         q += (long long)gridDim.x * blockDim.x)
      bdt_instance<LD_CA>(a.I[q]);
    if (!grid_sync(a.bar, a.expected, a.status, a.limit_ns)) return;
    for (int l = 0; l < a.stages; ++l) {
      const double ca = BSSP3_CA[l];
      for (long long b = blockIdx.x; b < a.ntiles; b += gridDim.x)
        bstage_tile<SYS, BC, R, LD_CA>(a.I, a.n, b, l, ca, 1.0 - ca, smem);
      if (!grid_sync(a.bar, a.expected, a.status, a.limit_ns)) return;
      const int nw = blockDim.x >> 5;
      for (long long it = (long long)blockIdx.x * nw + (threadIdx.x >> 5); it < (long long)a.n * 2 * F;
           it += (long long)gridDim.x * nw) {
        const BatchInst& in = a.I[it / (2 * F)];
        const int mesh = (int)((it / F) & 1), f = (int)(it % F);
        warp_sigma<LD_CA>(in.part, (long long)in.tx * in.ty, F, mesh, f, plain_norm(in.g.plane), in.avg, in.sigma);
      }
      if (!grid_sync(a.bar, a.expected, a.status, a.limit_ns)) return;
      for (long long b = blockIdx.x; b < a.ntiles; b += gridDim.x) {
        __syncthreads();  // the previous tile's readers of isg are done
        boe_tile<SYS, BC, R, LD_CA, false>(a.I, a.n, b, l == 2, isg, a.status);
      }
      if (!grid_sync(a.bar, a.expected, a.status, a.limit_ns)) return;
    }
  }
}

__global__ void k_bset_time(const BatchInst* __restrict__ I, int n, double t) {
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q < n) I[q].time[0] = t;
}

}  // namespace oecdg

using namespace oecdg;

struct cdg_batch {
  int n;
  int F;
  int sys, bc;
  int rows;                // tile height R in use
  cudaStream_t stream;
  int own_stream;
  BatchInst* h_inst;       // host copy of the instance table
  BatchInst* d_inst;       // device instance table
  long long total_blocks;  // stage and OE grid size for `rows`
  double* pool;            // one allocation: scratch states + partials + small slots
  int* status;
  double** h_ptrs;         // the caller's state pointers last uploaded
  cudaGraphExec_t graph;
  int graph_steps;
  int graph_flags;         // the cdg_batch_step flags the graph was captured with
  long long launches;
  // persistent mode
  unsigned long long* bar; // grid-barrier arrival counter (device)
  int nsm;                 // SMs of the device
  int bps;                 // persistent blocks per SM (0: as many as fit)
  double wait_s;           // bounded wait of every grid barrier
  int withhold;            // test hook: arrivals every barrier waits for that never come
  char err[256];
};

static cdg_status bfail(cdg_batch* b, cdg_status s, const char* msg) {
  if (b) snprintf(b->err, sizeof b->err, "%s", msg);
  return s;
}

// The instance table to the device, after everything already issued to the
// legacy default stream.  The copy is complete on return: a plain cudaMemcpy from
// pageable memory may come back before its DMA has reached the device, and a
// batch stream that does not wait for the legacy stream could then start its
// kernels on the old table (a null or stale state pointer).
static cudaError_t upload_table(cdg_batch* B) {
  const cudaError_t e = cudaMemcpy(B->d_inst, B->h_inst, sizeof(BatchInst) * B->n, cudaMemcpyHostToDevice);
  return e != cudaSuccess ? e : cudaStreamSynchronize(cudaStreamLegacy);
}

// tile table for tile height R; uploads the instance table
static cudaError_t batch_layout(cdg_batch* B, int R) {
  long long blk = 0;
  for (int q = 0; q < B->n; ++q) {
    BatchInst& in = B->h_inst[q];
    in.tx = (in.g.nx + SW_CELLS - 1) / SW_CELLS;
    in.ty = (in.g.ny + R - 1) / R;
    in.blk0 = blk;
    blk += 2LL * in.tx * in.ty;
  }
  B->total_blocks = blk;
  B->rows = R;
  if (B->graph) {
    cudaGraphExecDestroy(B->graph);
    B->graph = nullptr;
    B->graph_steps = 0;
  }
  return upload_table(B);
}

template <int SYS, int R>
constexpr int stage_smem() { return R * StageSmem<SYS>::WARP * (int)sizeof(double); }

template <int SYS, int BC, int R>
static cudaError_t launch_bstage_r(cdg_batch* B, int l, double ca, double cb) {
  constexpr int smem = stage_smem<SYS, R>();
  const cudaError_t e =
      cudaFuncSetAttribute(k_bstage<SYS, BC, R>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  k_bstage<SYS, BC, R><<<(unsigned)B->total_blocks, 32 * R, smem, B->stream>>>(B->d_inst, B->n, l, ca, cb);
  return cudaGetLastError();
}

template <int SYS, int BC>
static cudaError_t launch_bstage_t(cdg_batch* B, int l, double ca, double cb) {
  switch (B->rows) {
    case 2: return launch_bstage_r<SYS, BC, 2>(B, l, ca, cb);
    case 8: return launch_bstage_r<SYS, BC, 8>(B, l, ca, cb);
    default: return launch_bstage_r<SYS, BC, 4>(B, l, ca, cb);
  }
}

template <int SYS, int BC, bool SQUARE>
static cudaError_t launch_boe_t(cdg_batch* B, int last) {
  const unsigned grid = (unsigned)B->total_blocks;
  switch (B->rows) {
    case 2: k_boe<SYS, BC, 2, SQUARE><<<grid, 64, 0, B->stream>>>(B->d_inst, B->n, last, B->status); break;
    case 8: k_boe<SYS, BC, 8, SQUARE><<<grid, 256, 0, B->stream>>>(B->d_inst, B->n, last, B->status); break;
    default: k_boe<SYS, BC, 4, SQUARE><<<grid, 128, 0, B->stream>>>(B->d_inst, B->n, last, B->status); break;
  }
  return cudaGetLastError();
}

static cudaError_t launch_bstage(cdg_batch* B, int l, double ca, double cb) {
  B->launches += 1;
  if (B->bc == BC_PERIODIC) return launch_bstage_t<SYS_EULER, BC_PERIODIC>(B, l, ca, cb);
  return launch_bstage_t<SYS_EULER, BC_TRANSMISSIVE>(B, l, ca, cb);
}

static cudaError_t launch_boe(cdg_batch* B, int last) {
  B->launches += 1;
  bool square = true;
  for (int q = 0; q < B->n; ++q) square = square && oe_form(B->h_inst[q].g) == OE_SQUARE;
  if (B->bc == BC_PERIODIC)
    return square ? launch_boe_t<SYS_EULER, BC_PERIODIC, true>(B, last)
                  : launch_boe_t<SYS_EULER, BC_PERIODIC, false>(B, last);
  return square ? launch_boe_t<SYS_EULER, BC_TRANSMISSIVE, true>(B, last)
                : launch_boe_t<SYS_EULER, BC_TRANSMISSIVE, false>(B, last);
}

static const double BSSP3_C[3] = {0.0, 0.75, 1.0 / 3.0};

// one SSP-RK3 step of every instance: 11 launches
static cudaError_t batch_one_step(cdg_batch* B) {
  k_bwave<SYS_EULER><<<dim3(WB, B->n), 256, 0, B->stream>>>(B->d_inst, B->status);
  k_bdt<<<(B->n + 127) / 128, 128, 0, B->stream>>>(B->d_inst, B->n);
  B->launches += 2;
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  for (int l = 0; l < 3; ++l) {
    const double ca = BSSP3_C[l];
    if ((e = launch_bstage(B, l, ca, 1.0 - ca)) != cudaSuccess) return e;
    k_bsigma<<<dim3(B->F, 2, B->n), 32, 0, B->stream>>>(B->d_inst, B->F);
    B->launches += 1;
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    if ((e = launch_boe(B, l == 2)) != cudaSuccess) return e;
  }
  return cudaSuccess;
}

// Blocks per SM of the persistent kernel that fit (and its shared memory limit).
template <int BC, int R>
static cudaError_t bpersist_occupancy_t(int* occ) {
  auto kern = k_bpersist<SYS_EULER, BC, R>;
  constexpr int smem = stage_smem<SYS_EULER, R>();
  const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(occ, kern, 32 * R, smem);
}

// One cooperative launch of nsteps steps (`stages` stages each, see
// BPersistArgs); the arrival counter is zeroed first (a memset node when
// captured).  Grid: blocks per SM x SMs, at most what fits and at most the
// tiles.
template <int BC, int R>
static cudaError_t launch_bpersist_t(cdg_batch* B, int nsteps, int stages, long long* grid_out) {
  auto kern = k_bpersist<SYS_EULER, BC, R>;
  int occ = 0;
  cudaError_t e = bpersist_occupancy_t<BC, R>(&occ);
  if (e != cudaSuccess) return e;
  if (occ < 1) return cudaErrorCooperativeLaunchTooLarge;
  const int bps = (B->bps > 0 && B->bps < occ) ? B->bps : occ;
  long long grid = (long long)bps * B->nsm;
  if (grid > B->total_blocks) grid = B->total_blocks;
  if (grid_out) *grid_out = grid;
  BPersistArgs a;
  a.I = B->d_inst;
  a.n = B->n;
  a.ntiles = B->total_blocks;
  a.nsteps = nsteps;
  a.bar = B->bar;
  a.expected = (unsigned long long)grid + (unsigned long long)B->withhold;
  a.limit_ns = (unsigned long long)(B->wait_s * 1e9);
  a.status = B->status;
  a.stages = stages;
  if ((e = cudaMemsetAsync(B->bar, 0, sizeof(unsigned long long), B->stream)) != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3(32 * R);
  cfg.dynamicSmemBytes = stage_smem<SYS_EULER, R>();
  cfg.stream = B->stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, a);
}

template <int BC>
static cudaError_t launch_bpersist_bc(cdg_batch* B, int nsteps, int stages, long long* grid) {
  switch (B->rows) {
    case 2: return launch_bpersist_t<BC, 2>(B, nsteps, stages, grid);
    case 8: return launch_bpersist_t<BC, 8>(B, nsteps, stages, grid);
    default: return launch_bpersist_t<BC, 4>(B, nsteps, stages, grid);
  }
}

static cudaError_t launch_bpersist(cdg_batch* B, int nsteps, int stages, long long* grid = nullptr) {
  B->launches += 1;
  if (B->bc == BC_PERIODIC) return launch_bpersist_bc<BC_PERIODIC>(B, nsteps, stages, grid);
  return launch_bpersist_bc<BC_TRANSMISSIVE>(B, nsteps, stages, grid);
}

// blocks per SM of the persistent kernel that fit for tile height R
static int persist_occupancy(const cdg_batch* B, int R) {
  int occ = 0;
  cudaError_t e;
  if (B->bc == BC_PERIODIC)
    e = R == 2   ? bpersist_occupancy_t<BC_PERIODIC, 2>(&occ)
        : R == 8 ? bpersist_occupancy_t<BC_PERIODIC, 8>(&occ)
                 : bpersist_occupancy_t<BC_PERIODIC, 4>(&occ);
  else
    e = R == 2   ? bpersist_occupancy_t<BC_TRANSMISSIVE, 2>(&occ)
        : R == 8 ? bpersist_occupancy_t<BC_TRANSMISSIVE, 8>(&occ)
                 : bpersist_occupancy_t<BC_TRANSMISSIVE, 4>(&occ);
  return e == cudaSuccess ? occ : 0;
}

extern "C" {

cdg_status cdg_init_batch(const cdg_mesh_desc* descs, int n, void* stream, cdg_batch** out) {
  if (out) *out = nullptr;
  if (!descs || !out || n < 1) return CDG_EINVAL;
  for (int q = 0; q < n; ++q) {
    const cdg_mesh_desc& d = descs[q];
    if (d.dim != 2 || d.nx < 2 || d.ny < 2) return CDG_EINVAL;
    if (d.system != CDG_EULER || d.k != 2 || d.basis != CDG_BASIS_Q || d.rk != CDG_RK_SSP3 || d.oe != 1)
      return CDG_EUNSUPPORTED;
    if (invalid_sides(d) || uniform_side_bc(d) < 0) return CDG_EINVAL;
    if (uniform_side_bc(d) != uniform_side_bc(descs[0])) return CDG_EINVAL;
    if (!(d.bx > d.ax) || !(d.by > d.ay) || !(d.cfl > 0.0) || !(d.gamma > 1.0)) return CDG_EINVAL;
  }
  cdg_batch* B = (cdg_batch*)calloc(1, sizeof(cdg_batch));
  if (!B) return CDG_ENOMEM;
  B->n = n;
  B->F = 4;
  B->sys = SYS_EULER;
  B->bc = uniform_side_bc(descs[0]) == CDG_PERIODIC ? BC_PERIODIC : BC_TRANSMISSIVE;
  B->h_inst = (BatchInst*)calloc(n, sizeof(BatchInst));
  B->h_ptrs = (double**)calloc(n, sizeof(double*));
  if (!B->h_inst || !B->h_ptrs) {
    cdg_batch_free(B);
    return CDG_ENOMEM;
  }
  if (stream) {
    B->stream = (cudaStream_t)stream;
  } else {
    if (cudaStreamCreateWithFlags(&B->stream, cudaStreamNonBlocking) != cudaSuccess) {
      cdg_batch_free(B);
      return CDG_ECUDA;
    }
    B->own_stream = 1;
  }
  // pool: per instance 2 scratch states, partials for the smallest tile height
  // (the most tiles), wave partials and the small slots
  size_t total = 0;
  for (int q = 0; q < n; ++q) {
    const cdg_mesh_desc& d = descs[q];
    const size_t plane = (size_t)d.nx * d.ny;
    const size_t tiles = (size_t)((d.nx + SW_CELLS - 1) / SW_CELLS) * ((d.ny + 1) / 2);
    total += 2 * (size_t)2 * 4 * 9 * plane + 2 * tiles * 4 * 3 + WB * 2 + 2 + 2 + 8 + 8;
  }
  B->wait_s = 5.0;
  {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&B->nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
      cdg_batch_free(B);
      return CDG_ECUDA;
    }
  }
  if (cudaMalloc((void**)&B->pool, total * sizeof(double)) != cudaSuccess ||
      cudaMalloc((void**)&B->d_inst, sizeof(BatchInst) * n) != cudaSuccess ||
      cudaMalloc((void**)&B->status, sizeof(int)) != cudaSuccess ||
      cudaMalloc((void**)&B->bar, sizeof(unsigned long long)) != cudaSuccess) {
    (void)cudaGetLastError();  // clear the failed allocation: later launch checks must not see it
    cdg_batch_free(B);
    return CDG_ENOMEM;
  }
  double* p = B->pool;
  for (int q = 0; q < n; ++q) {
    const cdg_mesh_desc& d = descs[q];
    BatchInst& in = B->h_inst[q];
    Geo& g = in.g;
    g.nx = d.nx;
    g.ny = d.ny;
    geo_sides(d, g);  // uniform periodic or transmissive: no padding
    g.hx = (d.bx - d.ax) / d.nx;
    g.hy = (d.by - d.ay) / d.ny;
    g.gamma = d.gamma;
    g.adv_x = d.adv_x;
    g.adv_y = d.adv_y;
    g.cfl = d.cfl;
    finish_geo(g);
    const size_t st = (size_t)2 * 4 * 9 * g.plane;
    const size_t tiles = (size_t)((d.nx + SW_CELLS - 1) / SW_CELLS) * ((d.ny + 1) / 2);
    in.a = p; p += st;
    in.b = p; p += st;
    in.part = p; p += 2 * tiles * 4 * 3;
    in.wpart = p; p += WB * 2;
    in.dt = p; p += 2;
    in.time = p; p += 2;
    in.sigma = p; p += 8;
    in.avg = p; p += 8;
    in.u = nullptr;
  }
  if (batch_layout(B, 4) != cudaSuccess || cudaMemsetAsync(B->status, 0, sizeof(int), B->stream) != cudaSuccess) {
    cdg_batch_free(B);
    return CDG_ECUDA;
  }
  k_bset_time<<<(n + 127) / 128, 128, 0, B->stream>>>(B->d_inst, n, 0.0);
  if (cudaGetLastError() != cudaSuccess || cudaStreamSynchronize(B->stream) != cudaSuccess) {
    cdg_batch_free(B);
    return CDG_ECUDA;
  }
  *out = B;
  return CDG_OK;
}

cdg_status cdg_batch_free(cdg_batch* B) {
  if (!B) return CDG_OK;
  if (B->stream) cudaStreamSynchronize(B->stream);
  if (B->graph) cudaGraphExecDestroy(B->graph);
  cudaFree(B->pool);
  cudaFree(B->d_inst);
  cudaFree(B->status);
  cudaFree(B->bar);
  if (B->own_stream) cudaStreamDestroy(B->stream);
  free(B->h_inst);
  free(B->h_ptrs);
  free(B);
  return CDG_OK;
}

const char* cdg_batch_last_error(const cdg_batch* B) { return B ? B->err : ""; }

// point the instance table at the caller's states (re-uploads only on change)
static cdg_status batch_bind(cdg_batch* B, double* const* d_us) {
  int changed = 0;
  for (int q = 0; q < B->n; ++q) {
    if (!d_us[q]) return bfail(B, CDG_EINVAL, "batch: null state pointer");
    if (B->h_ptrs[q] != d_us[q]) changed = 1;
  }
  if (!changed) return CDG_OK;
  for (int q = 0; q < B->n; ++q) {
    B->h_ptrs[q] = d_us[q];
    B->h_inst[q].u = d_us[q];
  }
  if (B->graph) {
    cudaGraphExecDestroy(B->graph);
    B->graph = nullptr;
    B->graph_steps = 0;
  }
  if (cudaStreamSynchronize(B->stream) != cudaSuccess || upload_table(B) != cudaSuccess)
    return bfail(B, CDG_ECUDA, "batch: uploading the instance table failed");
  return CDG_OK;
}

cdg_status cdg_batch_step(cdg_batch* B, double* const* d_us, int nsteps, int flags) {
  if (!B || !d_us || nsteps < 0 || flags < 0 || flags > 3) return bfail(B, CDG_EINVAL, "batch_step: bad arguments");
  cdg_status s = batch_bind(B, d_us);
  if (s != CDG_OK) return s;
  if (nsteps == 0) return CDG_OK;
  const int use_graph = flags & CDG_BATCH_GRAPH, persist = flags & CDG_BATCH_PERSISTENT;
  if (!use_graph) {
    if (persist) {
      if (launch_bpersist(B, nsteps, 3) != cudaSuccess) return bfail(B, CDG_ECUDA, "batch_step: persistent launch failed");
      return CDG_OK;
    }
    for (int k = 0; k < nsteps; ++k)
      if (batch_one_step(B) != cudaSuccess) return bfail(B, CDG_ECUDA, "batch_step: launch failed");
    return CDG_OK;
  }
  if (!B->graph || B->graph_steps != nsteps || B->graph_flags != flags) {
    if (B->graph) {
      cudaGraphExecDestroy(B->graph);
      B->graph = nullptr;
    }
    cudaGraph_t graph;
    if (cudaStreamBeginCapture(B->stream, cudaStreamCaptureModeThreadLocal) != cudaSuccess)
      return bfail(B, CDG_ECUDA, "batch_step: stream capture failed to begin");
    cudaError_t e = cudaSuccess;
    const long long before = B->launches;  // captured launches are counted when the graph runs
    if (persist) e = launch_bpersist(B, nsteps, 3);
    else
      for (int k = 0; k < nsteps && e == cudaSuccess; ++k) e = batch_one_step(B);
    B->launches = before;
    cudaError_t e2 = cudaStreamEndCapture(B->stream, &graph);
    if (e != cudaSuccess || e2 != cudaSuccess) return bfail(B, CDG_ECUDA, "batch_step: capture failed");
    e = cudaGraphInstantiate(&B->graph, graph, 0);
    cudaGraphDestroy(graph);
    if (e != cudaSuccess) return bfail(B, CDG_ECUDA, "batch_step: graph instantiation failed");
    B->graph_steps = nsteps;
    B->graph_flags = flags;
  }
  if (cudaGraphLaunch(B->graph, B->stream) != cudaSuccess) return bfail(B, CDG_ECUDA, "batch_step: graph launch failed");
  B->launches += persist ? 1 : 11LL * nsteps;
  return CDG_OK;
}

cdg_status cdg_batch_set_wait(cdg_batch* B, double limit_s, int withheld) {
  if (!B || !(limit_s > 0.0) || limit_s > 3600.0 || withheld < 0) return bfail(B, CDG_EINVAL, "batch_set_wait: bad arguments");
  if (cudaStreamSynchronize(B->stream) != cudaSuccess) return CDG_ECUDA;
  B->wait_s = limit_s;
  B->withhold = withheld;
  if (B->graph) {  // the limits are baked into a captured launch
    cudaGraphExecDestroy(B->graph);
    B->graph = nullptr;
    B->graph_steps = 0;
  }
  return CDG_OK;
}

cdg_status cdg_batch_set_grid(cdg_batch* B, int blocks_per_sm) {
  if (!B || blocks_per_sm < 0) return bfail(B, CDG_EINVAL, "batch_set_grid: bad arguments");
  if (cudaStreamSynchronize(B->stream) != cudaSuccess) return CDG_ECUDA;
  B->bps = blocks_per_sm;
  if (B->graph) {
    cudaGraphExecDestroy(B->graph);
    B->graph = nullptr;
    B->graph_steps = 0;
  }
  return CDG_OK;
}

cdg_status cdg_batch_grid(const cdg_batch* B, int* blocks_per_sm, int* grid) {
  if (!B || !blocks_per_sm || !grid) return CDG_EINVAL;
  const int occ = persist_occupancy(B, B->rows);
  if (occ < 1) return CDG_ECUDA;
  const int bps = (B->bps > 0 && B->bps < occ) ? B->bps : occ;
  long long g = (long long)bps * B->nsm;
  if (g > B->total_blocks) g = B->total_blocks;
  *blocks_per_sm = bps;
  *grid = (int)g;
  return CDG_OK;
}

cdg_status cdg_batch_check_status(cdg_batch* B) {
  if (!B) return CDG_EINVAL;
  int h = 0;
  if (cudaMemcpyAsync(&h, B->status, sizeof(int), cudaMemcpyDeviceToHost, B->stream) != cudaSuccess ||
      cudaMemsetAsync(B->status, 0, sizeof(int), B->stream) != cudaSuccess ||
      cudaStreamSynchronize(B->stream) != cudaSuccess)
    return bfail(B, CDG_ECUDA, "batch_check_status: CUDA error");
  if (h & ST_TIMEOUT) return bfail(B, CDG_ETIMEOUT, "a grid barrier of the persistent kernel ran out of time");
  if (h & ST_NONPHYSICAL) return bfail(B, CDG_ENONPHYSICAL, "non-physical cell average in the batch");
  return CDG_OK;
}

cdg_status cdg_batch_get_time(cdg_batch* B, double* t) {
  if (!B || !t) return CDG_EINVAL;
  if (cudaStreamSynchronize(B->stream) != cudaSuccess) return CDG_ECUDA;
  for (int q = 0; q < B->n; ++q)
    if (cudaMemcpy(t + q, B->h_inst[q].time, sizeof(double), cudaMemcpyDeviceToHost) != cudaSuccess) return CDG_ECUDA;
  return CDG_OK;
}

cdg_status cdg_batch_launch_count(const cdg_batch* B, long long* count) {
  if (!B || !count) return CDG_EINVAL;
  *count = B->launches;
  return CDG_OK;
}

cdg_status cdg_batch_set_rows(cdg_batch* B, int rows) {
  if (!B || (rows != 2 && rows != 4 && rows != 8)) return CDG_EINVAL;
  if (cudaStreamSynchronize(B->stream) != cudaSuccess || batch_layout(B, rows) != cudaSuccess) return CDG_ECUDA;
  return CDG_OK;
}

cdg_status cdg_batch_rows(const cdg_batch* B, int* rows) {
  if (!B || !rows) return CDG_EINVAL;
  *rows = B->rows;
  return CDG_OK;
}

// Signature of a batch for the autotune cache: the kernels' generation, sizes, boundary and
// count.  The generation (fx1: fixed point, tiles 8 cells wide) is raised with every change
// of what a choice of rows and grid stands for, so that a file tuned before is not used.
static void batch_signature(const cdg_batch* B, char* sig, size_t len) {
  unsigned long long h = 1469598103934665603ULL;
  for (int q = 0; q < B->n; ++q) {
    h = (h ^ (unsigned long long)B->h_inst[q].g.nx) * 1099511628211ULL;
    h = (h ^ (unsigned long long)B->h_inst[q].g.ny) * 1099511628211ULL;
  }
  snprintf(sig, len, "euler_q2_fx1_bc%d_n%d_%016llx", B->bc, B->n, h);
}

static int cache_lookup(const char* path, const char* sig) {
  FILE* f = fopen(path, "r");
  if (!f) return 0;
  char buf[1 << 16];
  size_t m = fread(buf, 1, sizeof buf - 1, f);
  fclose(f);
  buf[m] = 0;
  char key[160];
  snprintf(key, sizeof key, "\"%s\": ", sig);
  const char* p = strstr(buf, key);
  if (!p) return 0;
  return atoi(p + strlen(key));
}

static void cache_store(const char* path, const char* sig, int rows) {
  char buf[1 << 16];
  buf[0] = 0;
  FILE* f = fopen(path, "r");
  size_t m = 0;
  if (f) {
    m = fread(buf, 1, sizeof buf - 1, f);
    fclose(f);
  }
  buf[m] = 0;
  // keep previous entries: strip the closing brace of an existing object
  char* end = strrchr(buf, '}');
  f = fopen(path, "w");
  if (!f) return;
  if (end && strchr(buf, '{')) {
    *end = 0;
    char* last = end;
    while (last > buf && (last[-1] == ' ' || last[-1] == '\n')) --last;
    *last = 0;
    const int empty = last > buf && last[-1] == '{';
    fprintf(f, "%s%s\n  \"%s\": %d\n}\n", buf, empty ? "" : ",", sig, rows);
  } else {
    fprintf(f, "{\n  \"%s\": %d\n}\n", sig, rows);
  }
  fclose(f);
}

cdg_status cdg_batch_autotune(cdg_batch* B, double* const* d_us, const char* cache_path, int* rows_out) {
  if (!B || !d_us) return CDG_EINVAL;
  cdg_status s = batch_bind(B, d_us);
  if (s != CDG_OK) return s;
  char sig[128];
  batch_signature(B, sig, sizeof sig);
  // cache code: rows * 100 + blocks per SM (a bare 2, 4 or 8: rows only)
  const int code = cache_path ? cache_lookup(cache_path, sig) : 0;
  int best_rows = 0, best_bps = 0;
  if (code == 2 || code == 4 || code == 8) {
    best_rows = code;
  } else if (code >= 100) {
    const int r = code / 100, b = code % 100;
    if ((r == 2 || r == 4 || r == 8) && b >= 0 && b <= persist_occupancy(B, r)) {
      best_rows = r;
      best_bps = b;
    }
  }
  if (!best_rows) {
    // time the persistent kernel on one first stage of every instance (wave
    // speeds, tau, stage, sigma, OE into scratch: the caller's states are only
    // read) for every tile height and every persistent grid that fits; best of
    // two after a warm-up
    float best_ms = 1e30f;
    cudaEvent_t e0, e1;
    if (cudaEventCreate(&e0) != cudaSuccess || cudaEventCreate(&e1) != cudaSuccess) return CDG_ECUDA;
    const int saved_bps = B->bps;
    const int cand[3] = {2, 4, 8};
    for (int c = 0; c < 3; ++c) {
      if (batch_layout(B, cand[c]) != cudaSuccess) return CDG_ECUDA;
      const int occ = persist_occupancy(B, cand[c]);
      for (int bps = 1; bps <= occ; ++bps) {
        B->bps = bps;
        for (int rep = 0; rep < 3; ++rep) {
          cudaEventRecord(e0, B->stream);
          if (launch_bpersist(B, 1, 1) != cudaSuccess) return bfail(B, CDG_ECUDA, "autotune: launch failed");
          cudaEventRecord(e1, B->stream);
          if (cudaEventSynchronize(e1) != cudaSuccess) return bfail(B, CDG_ECUDA, "autotune: kernel failed");
          float ms = 0.f;
          cudaEventElapsedTime(&ms, e0, e1);
          if (rep > 0 && ms < best_ms) {
            best_ms = ms;
            best_rows = cand[c];
            best_bps = bps;
          }
        }
      }
    }
    B->bps = saved_bps;
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    k_bset_time<<<(B->n + 127) / 128, 128, 0, B->stream>>>(B->d_inst, B->n, 0.0);
    B->launches += 1;
    int h = 0;  // a timed-out candidate leaves its bit: report it rather than a choice
    if (cudaMemcpy(&h, B->status, sizeof(int), cudaMemcpyDeviceToHost) != cudaSuccess) return CDG_ECUDA;
    if (h & ST_TIMEOUT) return bfail(B, CDG_ETIMEOUT, "autotune: a grid barrier ran out of time");
    if (cache_path) cache_store(cache_path, sig, best_rows * 100 + best_bps);
  }
  if (batch_layout(B, best_rows) != cudaSuccess) return CDG_ECUDA;
  B->bps = best_bps;
  if (rows_out) *rows_out = best_rows;
  return CDG_OK;
}

}  // extern "C"
