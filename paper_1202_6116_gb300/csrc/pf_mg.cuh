// What the multigrid kernels share: smoothing weights and level diagonals.
#pragma once

#include "pf_internal.h"

namespace pf {

template <typename T>
__device__ __forceinline__ T mg_omega1() {
  return T(MG_OMEGA1);
}
template <typename T>
__device__ __forceinline__ T mg_omega2() {
  return T(MG_OMEGA2);
}

// 1/diag of a level's operator at column xy of plane z.
template <typename T>
__device__ __forceinline__ T mg_inv(const MgView<T>& L, int xy, int z) {
  if (L.g.periodic_z || (z > 0 && z < L.g.nz - 1)) return L.k.tab[0];
  return L.k.tab[3 * (z > 0 ? 0 : 1 + (int)L.tlo[xy]) + (z < L.g.nz - 1 ? 0 : 1 + (int)L.thi[xy])];
}

}  // namespace pf
