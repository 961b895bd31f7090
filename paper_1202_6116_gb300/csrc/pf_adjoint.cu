// Discrete adjoint of one forward-Euler TDGL step (Eq. TDGL with Eqs. F_bulk,
// dF_grad/dP, F_elec, rho and Poisson; Section Time Integration).
//
// The forward step is P' = P + dt L (-f'(P) + g Lap P + E(phi)), with
// A phi = -div P + B(V).  The face rules make the zero-voltage field operator
// E0 the transpose of div, and A and Lap are symmetric, so for a cotangent
// lam = dJ/dP' the transposed step is
//   lam_out = lam + dt L (-H(P) lam + g Lap lam + E0(psi)),  A psi = -div lam,
// H the 3x3 Hessian of the Landau density at each cell.  The adjoint
// potential psi comes from the same right-hand-side and Krylov kernels as the
// forward potential, run with the electrode voltages at zero; this file holds
// the update kernel, which also reduces the step's parameter sensitivities
//   d/da1  : -dt L sum lam . 2P
//   d/da11 : -dt L sum lam . 4P^3
//   d/da12 : -dt L sum lam_i 2P_i (P_j^2 + P_k^2)
//   d/dg   :  dt L sum lam . Lap P  (= dt L sum P . Lap lam, Lap symmetric)
// and, at every electrode face cell, the voltage sensitivity
//   bottom:  dt L (-psi_c 2 eps_c / dx^2 + lam_z,c / dx)
//   top:     dt L (-psi_c 2 eps_c / dx^2 - lam_z,c / dx).
// Algorithmic traffic per cell: reads lam (3), psi (1), P (3); writes lam_out (3).
#include "pf_internal.h"
#include "pf_march.cuh"

namespace pf {

constexpr int ADJ_D = 2;
constexpr int ADJ_NV = 4;

template <typename T, int VX>
using AdjPipe = Pipe<T, void, MTX, MTY, VX, 4, 3, ADJ_D>;

// The Hessian's and the stencils' factors (formed in FP64, rounded once) and, apart
// from them as in the forward update, dt L.
template <typename T>
struct AdjCoef {
  T h1, h11, h12, hx;            // -2 a1, -12 a11, -2 a12, -4 a12
  T gl, el;                      // g/dx^2, -1/(2 dx)
  T m;                           // dt L
  double dtL;
};

template <typename T>
struct L3 {
  T x, y, z;
};

template <typename T, int VX>
__global__ void __launch_bounds__(MTX* MTY) k_tdgl_adj(Geo g, Bc<T> bc, const T* __restrict__ lam,
                                                      T* __restrict__ lam_out, const T* __restrict__ psi,
                                                      const T* __restrict__ P, const T* __restrict__ eps,
                                                      AdjCoef<T> k, double* __restrict__ grad,
                                                      double* __restrict__ gv_lo, double* __restrict__ gv_hi,
                                                      double* part, Scalars* S, MarchCfg mc) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ long long tile_slot;
  const T* hsrc[4] = {lam, lam + g.n, lam + 2 * g.n, psi};
  const T* osrc[3] = {P, P + g.n, P + 2 * g.n};
  Acc<T> acc[ADJ_NV];
  TileGeo<MTX, MTY, VX> s{};
  auto emit = [&](int xy, int z, const Stencil7<Raw<T, 4>>& st, const T (&o)[3], const bool bt) -> L3<T> {
    // E0(psi): face values with every electrode at 0 V (doubled, as in tdgl_inc)
    const T fc = st.c.v[3];
    T dpsi[3];
    dpsi[0] = st.xp.v[3] - st.xm.v[3];
    dpsi[1] = st.yp.v[3] - st.ym.v[3];
    if (st.zb >= 0 && st.za >= 0) {
      dpsi[2] = st.zp.v[3] - st.zm.v[3];
    } else {
      const T flo = st.zb >= 0 ? fc + st.zm.v[3] : (bc.tlo[xy] ? T(0) : T(2) * fc);
      const T fhi = st.za >= 0 ? fc + st.zp.v[3] : (bc.thi[xy] ? T(0) : T(2) * fc);
      dpsi[2] = fhi - flo;
    }
    const T p[3] = {o[0], o[1], o[2]};
    const T l[3] = {st.c.v[0], st.c.v[1], st.c.v[2]};
    // (H lam)_i = lam_i (2 a1 + 12 a11 P_i^2 + 2 a12 q_i) + 4 a12 P_i d_i with q_i the
    // sum of the other two P_j^2 and d_i that of the other two P_j lam_j; the products
    // serve the sensitivities too: 87 FP64 operations a cell where the terms written
    // out took 196.  (Sums over all three, less the own one, are four operations fewer
    // and round twice: in FP32 the quartic coefficient along an axis is 1e-7 off.)
    T p2[3], pl[3], out[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      p2[i] = p[i] * p[i];
      pl[i] = p[i] * l[i];
    }
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      const int j = (i + 1) % 3, q = (i + 2) % 3;
      T lap = st.xp.v[i] - l[i];
      lap -= l[i] - st.xm.v[i];
      lap += st.yp.v[i] - l[i];
      lap -= l[i] - st.ym.v[i];
      if (st.zb >= 0) lap += st.zm.v[i] - l[i];
      if (st.za >= 0) lap += st.zp.v[i] - l[i];
      const T pq = fma(p[j], p[j], p2[q]);
      const T Hl = fma(l[i], fma(k.h12, pq, fma(k.h11, p2[i], k.h1)), k.hx * p[i] * fma(p[j], l[j], pl[q]));
      out[i] = l[i] + k.m * (k.gl * lap + (k.el * dpsi[i] + Hl));
      acc[0].add(l[i], p[i]);
      acc[1].add(p2[i], pl[i]);
      acc[2].add(pl[i], pq);
      acc[3].add(p[i], lap);
    }
    if (bt) {
      const long long c = (long long)z * g.nxy + xy;
      const double dtL = k.dtL;
      const double ec = eps ? (double)eps[c] : 1.0;
      const double qpsi = -(double)fc * 2.0 * ec * g.ih2;
      if (gv_lo && st.zb < 0 && bc.tlo[xy]) gv_lo[xy] += dtL * (qpsi + (double)l[2] * g.ih);
      if (gv_hi && st.za < 0 && bc.thi[xy]) gv_hi[xy] += dtL * (qpsi - (double)l[2] * g.ih);
    }
    return L3<T>{out[0], out[1], out[2]};
  };
  auto post = [&](int z, const L3<T> (&ov)[VX]) {
#pragma unroll
    for (int q = 0; q < ADJ_NV; ++q) acc[q].run();
    const long long c = (long long)z * g.nxy + s.xy;
    T a[VX], b[VX], d[VX];
#pragma unroll
    for (int i = 0; i < VX; ++i) {
      a[i] = ov[i].x;
      b[i] = ov[i].y;
      d[i] = ov[i].z;
    }
    store_n<T, VX>(lam_out + c, a);
    store_n<T, VX>(lam_out + g.n + c, b);
    store_n<T, VX>(lam_out + 2 * g.n + c, d);
  };
  const TileSched ts{&S->sched_next, &S->sched_done, mc.ntiles};
  for (long long t = sched_first(ts, &tile_slot); t < mc.ntiles; t = sched_next(ts, &tile_slot)) {
    s = tile_geo<MTX, MTY, VX>(g, t, mc);
#pragma unroll
    for (int q = 0; q < ADJ_NV; ++q) acc[q] = Acc<T>();
    march_direct<T, L3<T>, MTX, MTY, VX, 4, 3, ADJ_D>(g, s, smem, hsrc, osrc, emit, post);
    typename SumOf<T>::type v[ADJ_NV];
#pragma unroll
    for (int q = 0; q < ADJ_NV; ++q) v[q] = acc[q].sum();
    tile_partials<ADJ_NV, MTX * MTY>(v, part, t, smem);
  }
  sched_finish(ts);
  if (!last_block<MTX * MTY>(&S->ticket)) return;
  double sum[ADJ_NV];
  gather_partials<ADJ_NV, MTX * MTY>(part, mc.ntiles, sum, smem);
  if (threadIdx.x != 0 || threadIdx.y != 0) return;
  const double dtL = k.dtL;
  grad[0] += -2.0 * dtL * sum[0];
  grad[1] += -4.0 * dtL * sum[1];
  grad[2] += -2.0 * dtL * sum[2];
  grad[3] += dtL * g.ih2 * sum[3];
  S->ticket = 0;
}

template <typename T, int VX>
static void adj_t(const LaunchCfg& L, const Geo& g, const Dev<T>& d, const T* lam, T* lam_out, const T* psi,
                  const T* P, const AdjCoef<T>& k, double* grad, double* gv_lo, double* gv_hi) {
  static bool once = false;
  const size_t bytes = AdjPipe<T, VX>::bytes();
  if (!once) {
    allow_smem(k_tdgl_adj<T, VX>, bytes);
    once = true;
  }
  static int occ = 0;
  const MarchCfg mc = kernel_tiling(k_tdgl_adj<T, VX>, bytes, L, occ, false);
  k_tdgl_adj<T, VX><<<mc.grid, dim3(MTX, MTY), bytes, L.stream>>>(
      g, d.bc, lam, lam_out, psi, P, d.eps, k, grad, gv_lo, gv_hi, d.part, d.S, mc);
}

template <typename T>
void launch_tdgl_adj(const LaunchCfg& L, const Geo& g, const Dev<T>& d, const T* lam, T* lam_out, const T* psi,
                     const T* P, const double* coef, double* grad, double* gv_lo, double* gv_hi) {
  const double dtL = coef[4];
  const AdjCoef<T> k{T(-2.0 * coef[0]),
                     T(-12.0 * coef[1]),
                     T(-2.0 * coef[2]),
                     T(-4.0 * coef[2]),
                     T(coef[3] * g.ih2),
                     T(-0.5 * g.ih),
                     T(dtL),
                     dtL};
  constexpr int V = 16 / sizeof(T);
  if (L.march.vx == V) adj_t<T, V>(L, g, d, lam, lam_out, psi, P, k, grad, gv_lo, gv_hi);
  else adj_t<T, 1>(L, g, d, lam, lam_out, psi, P, k, grad, gv_lo, gv_hi);
}

template void launch_tdgl_adj<float>(const LaunchCfg&, const Geo&, const Dev<float>&, const float*, float*,
                                     const float*, const float*, const double*, double*, double*, double*);
template void launch_tdgl_adj<double>(const LaunchCfg&, const Geo&, const Dev<double>&, const double*, double*,
                                      const double*, const double*, const double*, double*, double*, double*);

}  // namespace pf
