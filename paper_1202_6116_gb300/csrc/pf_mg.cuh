// What the multigrid kernels share: smoothing weights and level diagonals.
#pragma once

#include "pf_internal.h"

namespace pf {

// Jacobi weights of the two smoothing sweeps: the reciprocals of the roots of
// the degree-2 Chebyshev polynomial on [b/4, b], b = 1.9, which bound the
// spectrum of diag(A)^-1 A (in [0, 2] for this M-matrix) from below b/4 up,
// i.e. 1/lambda_k with lambda_k = (b + a)/2 + (b - a)/2 cos((2k - 1) pi / 4),
// a = b/4.  The pair damps the upper three quarters of the spectrum (the part
// the coarse grid cannot represent) by |(1 - w1 l)(1 - w2 l)| <= 0.35 on
// [b/4, 2]; weighted Jacobi with 6/7 twice leaves up to 0.51 there.  The
// pre-smoother applies w1 then w2, the post-smoother w2 then w1.
template <typename T>
__device__ __forceinline__ T mg_omega1() {
  return T(0.5912564121058501);
}
template <typename T>
__device__ __forceinline__ T mg_omega2() {
  return T(1.462658863889015);
}

// 1/diag of a level's operator at column xy of plane z.
template <typename T>
__device__ __forceinline__ T mg_inv(const MgView<T>& L, int xy, int z, T inv_int) {
  if (L.g.periodic_z || (z > 0 && z < L.g.nz - 1)) return inv_int;
  const int cz = (z > 0 ? 1 : 2 * (int)L.tlo[xy]) + (z < L.g.nz - 1 ? 1 : 2 * (int)L.thi[xy]);
  return T(1) / (T(2) * L.ax + T(2) * L.ay + T(cz) * L.az);
}

template <typename T>
__device__ __forceinline__ T mg_inv_int(const MgView<T>& L) {
  return T(1) / (T(2) * L.ax + T(2) * L.ay + T(2) * L.az);
}

}  // namespace pf
