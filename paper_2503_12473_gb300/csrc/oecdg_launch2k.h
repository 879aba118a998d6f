// oecdg_launch2k.h -- launch helpers of the degree-generic 2D kernels.
#pragma once

#include <type_traits>

#include "oecdg_common.cuh"

namespace oecdg {

template <int V>
using ICk = std::integral_constant<int, V>;

// fn(IC<SYS>, IC<BC>, IC<K>, IC<B>) for the runtime (sys, bc, k, basis)
template <class Fn>
static void by_sys_bc_k_b(int sys, int bc, int k, int basis, Fn&& fn) {
  auto kb = [&](auto S, auto Bc) {
    if (basis == BASIS_Q) {
      if (k == 1) fn(S, Bc, ICk<1>{}, ICk<BASIS_Q>{});
      else if (k == 2) fn(S, Bc, ICk<2>{}, ICk<BASIS_Q>{});
      else fn(S, Bc, ICk<3>{}, ICk<BASIS_Q>{});
    } else {
      if (k == 1) fn(S, Bc, ICk<1>{}, ICk<BASIS_P>{});
      else if (k == 2) fn(S, Bc, ICk<2>{}, ICk<BASIS_P>{});
      else fn(S, Bc, ICk<3>{}, ICk<BASIS_P>{});
    }
  };
  auto bb = [&](auto S) {
    if (bc == BC_PERIODIC) kb(S, ICk<BC_PERIODIC>{});
    else if (bc == BC_TRANSMISSIVE) kb(S, ICk<BC_TRANSMISSIVE>{});
    else kb(S, ICk<BC_GENERAL>{});
  };
  if (sys == SYS_EULER) bb(ICk<SYS_EULER>{});
  else if (sys == SYS_BURGERS) bb(ICk<SYS_BURGERS>{});
  else bb(ICk<SYS_ADV>{});
}

// Tiles of 8 x rows cells of both meshes' padded layout, row after row in gridDim.x
// (gridDim.y ends at 65535: 131070 rows of cells in tiles of 2), the two meshes'
// blocks of a tile adjacent.  At most 2^31 cells and 2^31 / 4 narrow tiles: int.
static unsigned grid2k(const Geo& g, int rows) {
  return 2u * (unsigned)((g.nxs + 7) / 8) * (unsigned)((g.nys + rows - 1) / rows);
}

}  // namespace oecdg
