// The small levels of the multigrid V-cycle in one launch, and the coarsest
// level's inverse.
//
// A launch over a level of some ten thousand cells costs its latency, not its
// work: a 65 536-cell level took four launches of 4 to 5 us each for under a
// microsecond of memory traffic, and the levels below 4096 cells in one block
// 43 us (FP32) or 103 us (FP64, one SM's share of the FP64 unit).  k_mg_sub
// runs the whole V-cycle from the first level of at most mg_sub_cells() cells
// down and back up as one thread-block cluster:
//   wide levels    spread over the cluster's 16 blocks, fields in global memory
//                  (L2), a hardware cluster barrier between the phases;
//   solo levels    (at most mg_solo_cells(), where a barrier costs more than
//                  the idle SMs) in block 0, fields in its shared memory;
//   coarsest level the product with its inverse, a row per thread (small) or
//                  per warp over the cluster.
// Per level four phases: both pre-sweeps (the first formed on the fly),
// residual + restriction (a coarse cell per thread), prolongation sweep (e +
// P e_c formed on the fly), second post-sweep.  Operators, weights, transfers
// and face rules are those of the per-level kernels (pf_mg.cu).  When level 0
// is itself small the launch is the whole preconditioner and also forms r.z
// and beta.
//
// The coarsest operator changes only with the electrode layout, so its inverse
// is formed once per bind or layout change: in FP64, in place, one symmetric
// Gauss-Jordan step per unknown (the operator is positive definite, so no
// pivoting).  Conjugate gradients in one block, which this replaces, took
// 1.47 ms per V-cycle on a coarsest level of 567 cells (21 x 27 x 1): nine of
// its ten microseconds an iteration were FP64 reductions on one SM.
#include "pf_internal.h"
#include "pf_march.cuh"
#include "pf_mg.cuh"

namespace pf {

constexpr int SUB_CLUSTER = 16;
constexpr int SUB_ROWS = 64;      // coarsest levels up to this size: a row per thread of block 0

constexpr int SUB_THREADS = 512;

__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release;\nbarrier.cluster.wait.acquire;\n" ::: "memory");
}

// Quotient of a small non-negative int (a < 2^22) by d >= 1, r = 1 / d: the
// rounded product is at most one off, and one compare on each side corrects it.
__device__ __forceinline__ int small_div(int a, int d, float r) {
  int q = (int)((float)a * r);
  if (q * d > a) --q;
  else if ((q + 1) * d <= a) ++q;
  return q;
}

// Where a cell's diagonal stands in a level's tables.
template <typename T>
__device__ __forceinline__ int sub_kind(const SubDesc<T>& L, const int8_t* lo, const int8_t* hi, int x, int y, int z) {
  if (L.per || (z > 0 && z < L.nz - 1)) return 0;
  const int xy = y * L.nx + x;
  return 3 * (z > 0 ? 0 : 1 + (int)lo[xy]) + (z < L.nz - 1 ? 0 : 1 + (int)hi[xy]);
}

// 1/diag at cell (x, y, z) with linear index c; lo, hi: the level's face masks.
template <typename T, bool EPS>
__device__ __forceinline__ T sub_inv(const SubDesc<T>& L, const int8_t* lo, const int8_t* hi, int c, int x, int y,
                                     int z) {
  if constexpr (EPS) return L.invd[c];
  return L.tab[sub_kind(L, lo, hi, x, y, z)];
}

// VX cells in a row from (x, y, z) on: linear index, neighbour rows and planes
// (zm, zp < 0 past a face).
template <typename T, int VX>
struct SubRow {
  int x, y, z, c, ym, yp, zm, zp;
  // vector number i of the level
  __device__ __forceinline__ SubRow(const SubDesc<T>& L, int i) {
    const int nv = L.nx / VX, q = small_div(i, nv, VX * L.rnx);
    x = (i - q * nv) * VX;
    z = small_div(q, L.ny, L.rny);
    y = q - z * L.ny;
    around(L);
  }
  __device__ __forceinline__ SubRow(const SubDesc<T>& L, int x_, int y_, int z_) : x(x_), y(y_), z(z_) { around(L); }
  __device__ __forceinline__ void around(const SubDesc<T>& L) {
    c = (z * L.ny + y) * L.nx + x;
    ym = y == 0 ? L.ny - 1 : y - 1;
    yp = y == L.ny - 1 ? 0 : y + 1;
    zm = z > 0 ? z - 1 : (L.per ? L.nz - 1 : -1);
    zp = z < L.nz - 1 ? z + 1 : (L.per ? 0 : -1);
  }
};

// f - A v at VX cells in a row.  vec(index, x, y, z, o) gives v at the VX cells
// from there on, one(index, x, y, z) at one cell; vc: v at the cells
// themselves.  With eps = 1 as f - d v + S (d the diagonal, S the weighted sum
// of the neighbours): 7 FP64 operations a cell, 13 as differences.
template <typename T, bool EPS, int VX, class Vec, class One>
__device__ __forceinline__ void sub_res(const SubDesc<T>& L, const int8_t* lo, const int8_t* hi,
                                          const SubRow<T, VX>& s, const T (&fc)[VX], const T (&vc)[VX], T (&out)[VX],
                                        Vec vec, One one) {
  const int xl = s.x == 0 ? L.nx - 1 : s.x - 1, xr = s.x + VX == L.nx ? 0 : s.x + VX;
  const int cl = s.c - s.x + xl, cr = s.c - s.x + xr;
  const int cym = s.c + (s.ym - s.y) * L.nx, cyp = s.c + (s.yp - s.y) * L.nx;
  const int czm = s.c + (s.zm - s.z) * L.nxy, czp = s.c + (s.zp - s.z) * L.nxy;
  T ym[VX], yp[VX], zm[VX], zp[VX];
  const T vl = one(cl, xl, s.y, s.z), vr = one(cr, xr, s.y, s.z);
  vec(cym, s.x, s.ym, s.z, ym);
  vec(cyp, s.x, s.yp, s.z, yp);
#pragma unroll
  for (int i = 0; i < VX; ++i) zm[i] = zp[i] = T(0);
  if (s.zm >= 0) vec(czm, s.x, s.y, s.zm, zm);
  if (s.zp >= 0) vec(czp, s.x, s.y, s.zp, zp);
  if constexpr (EPS) {
    const int xy = s.y * L.nx + s.x;
    T ec[VX], eym[VX], eyp[VX], ezm[VX], ezp[VX];
    load_n<T, VX>(L.eps + s.c, ec);
    load_n<T, VX>(L.eps + cym, eym);
    load_n<T, VX>(L.eps + cyp, eyp);
#pragma unroll
    for (int i = 0; i < VX; ++i) ezm[i] = ezp[i] = T(1);
    if (s.zm >= 0) load_n<T, VX>(L.eps + czm, ezm);
    if (s.zp >= 0) load_n<T, VX>(L.eps + czp, ezp);
    const T el = L.eps[cl], er = L.eps[cr];
#pragma unroll
    for (int i = 0; i < VX; ++i) {
      const T v = vc[i], e = ec[i];
      const T eb = i == 0 ? el : ec[i - 1], ea = i == VX - 1 ? er : ec[i + 1];
      const T vb = i == 0 ? vl : vc[i - 1], va = i == VX - 1 ? vr : vc[i + 1];
      if (s.zm >= 0 && s.zp >= 0 &&
          (eb == e) & (ea == e) & (eym[i] == e) & (eyp[i] == e) & (ezm[i] == e) & (ezp[i] == e)) {   // see one_eps
        out[i] = fc[i] - e * (L.ax * ((v - vb) - (va - v)) + L.ay * ((v - ym[i]) - (yp[i] - v)) +
                              L.az * ((v - zm[i]) - (zp[i] - v)));
        continue;
      }
      const T sx = hmean2(e, eb) * (v - vb) - hmean2(e, ea) * (va - v);
      const T sy = hmean2(e, eym[i]) * (v - ym[i]) - hmean2(e, eyp[i]) * (yp[i] - v);
      T sz = T(0);
      if (s.zm >= 0) sz += hmean2(e, ezm[i]) * (v - zm[i]);
      else if (lo[xy + i]) sz += T(2) * e * v;
      if (s.zp >= 0) sz += hmean2(e, ezp[i]) * (v - zp[i]);
      else if (hi[xy + i]) sz += T(2) * e * v;
      out[i] = fc[i] - (L.ax * sx + L.ay * sy + L.az * sz);
    }
  } else {
#pragma unroll
    for (int i = 0; i < VX; ++i) {
      T r = fc[i] - L.diag[sub_kind(L, lo, hi, s.x + i, s.y, s.z)] * vc[i];
      r += L.az * (zm[i] + zp[i]);
      r += L.ay * (ym[i] + yp[i]);
      out[i] = r + L.ax * ((i == 0 ? vl : vc[i - 1]) + (i == VX - 1 ? vr : vc[i + 1]));
    }
  }
}

// The phases of a level (masks lo, hi), over its vectors i0, i0 + stride, ...
// e1 = om1 f / diag, the first pre-sweep from zero: formed by the restriction
// that made f, or on the fly (FLY: the first level, whose f comes from another
// kernel).
template <typename T, bool EPS, bool FLY, int VX>
__device__ __forceinline__ void sub_pre(const SubDesc<T>& L, const int8_t* lo, const int8_t* hi, const T* f,
                                        const T* e1, T* e, int i0, int stride) {
  const T om1 = mg_omega1<T>(), om2 = mg_omega2<T>();
  for (int i = i0; i < L.n / VX; i += stride) {
    const SubRow<T, VX> s(L, i);
    T fc[VX], ec[VX], inv[VX], res[VX];
    load_n<T, VX>(f + s.c, fc);
#pragma unroll
    for (int k = 0; k < VX; ++k) inv[k] = sub_inv<T, EPS>(L, lo, hi, s.c + k, s.x + k, s.y, s.z);
    if constexpr (FLY) {
      const bool near = EPS || (!L.per && (s.z <= 1 || s.z >= L.nz - 2));   // else one diagonal all around
      auto w = [&](int j, int x, int y, int z) -> T {
        return om1 * (near ? sub_inv<T, EPS>(L, lo, hi, j, x, y, z) : L.tab[0]);
      };
#pragma unroll
      for (int k = 0; k < VX; ++k) ec[k] = om1 * inv[k] * fc[k];
      sub_res<T, EPS, VX>(
          L, lo, hi, s, fc, ec, res,
          [&](int j, int x, int y, int z, T (&o)[VX]) {
            load_n<T, VX>(f + j, o);
#pragma unroll
            for (int k = 0; k < VX; ++k) o[k] *= w(j + k, x + k, y, z);
          },
          [&](int j, int x, int y, int z) -> T { return w(j, x, y, z) * f[j]; });
    } else {
      load_n<T, VX>(e1 + s.c, ec);
      sub_res<T, EPS, VX>(
          L, lo, hi, s, fc, ec, res, [&](int j, int, int, int, T (&o)[VX]) { load_n<T, VX>(e1 + j, o); },
          [&](int j, int, int, int) -> T { return e1[j]; });
    }
#pragma unroll
    for (int k = 0; k < VX; ++k) ec[k] += om2 * inv[k] * res[k];
    store_n<T, VX>(e + s.c, ec);
  }
}

// Residual and restriction to the next level C (masks clo, chi), with e1
// there: fy fz threads per group of coarse cells, each a row of children (VX
// cells, or with VX = 1 the fx children of one coarse cell).
template <typename T, bool EPS, int VX>
__device__ __forceinline__ void sub_restrict(const SubDesc<T>& L, const int8_t* lo, const int8_t* hi, const T* f,
                                             const T* e, const SubDesc<T>& C, const int8_t* clo, const int8_t* chi,
                                             T* fc, T* e1c, int i0, int stride) {
  const T scale = L.scale;
  const int cv = VX == 1 ? 1 : VX / L.fx;                          // coarse cells of a group
  const int gs = L.fy * L.fz, sh = gs >> 1, total = C.n / cv * gs; // gs = 1, 2, 4: shift 0, 1, 2
  const int lane = threadIdx.x & 31, nv = C.nx / cv;
  const float rnv = cv * C.rnx;
  for (int i = i0; i - lane < total; i += stride) {                // whole warps
    T acc[VX];
#pragma unroll
    for (int k = 0; k < VX; ++k) acc[k] = T(0);
    const int grp = i >> sh, sub = i & (gs - 1);
    const int q = small_div(grp, nv, rnv), X = (grp - q * nv) * cv, Z = small_div(q, C.ny, C.rny), Y = q - Z * C.ny;
    if (i < total) {
      const int y = Y * L.fy + (L.fy == 2 ? sub & 1 : 0), z = Z * L.fz + (L.fz == 2 ? sub >> (L.fy - 1) : 0);
      auto res = [&](int x, T (&o)[VX]) {
        const SubRow<T, VX> s(L, x, y, z);
        T ec[VX], fv[VX];
        load_n<T, VX>(e + s.c, ec);
        load_n<T, VX>(f + s.c, fv);
        sub_res<T, EPS, VX>(
            L, lo, hi, s, fv, ec, o, [&](int j, int, int, int, T (&v)[VX]) { load_n<T, VX>(e + j, v); },
            [&](int j, int, int, int) -> T { return e[j]; });
      };
      res(X * L.fx, acc);
      if (L.fx == 2) {
        if constexpr (VX == 1) {
          T more[1];
          res(X * 2 + 1, more);
          acc[0] += more[0];
        } else {
#pragma unroll
          for (int k = 0; k < VX / 2; ++k) acc[k] = acc[2 * k] + acc[2 * k + 1];
        }
      }
    }
#pragma unroll
    for (int k = 0; k < VX; ++k) {
      if (gs > 1) acc[k] += __shfl_xor_sync(0xffffffffu, acc[k], 1);
      if (gs > 2) acc[k] += __shfl_xor_sync(0xffffffffu, acc[k], 2);
    }
    if (i < total && sub == 0) {
      const int cell = (Z * C.ny + Y) * C.nx + X;
#pragma unroll
      for (int k = 0; k < VX; ++k)
        if (k < cv) {
          const T v = acc[k] * scale;
          fc[cell + k] = v;
          e1c[cell + k] = mg_omega1<T>() * sub_inv<T, EPS>(C, clo, chi, cell + k, X + k, Y, Z) * v;
        }
    }
  }
}

template <typename T, bool EPS, int VX>
__device__ __forceinline__ void sub_post1(const SubDesc<T>& L, const int8_t* lo, const int8_t* hi, const T* f,
                                          const T* e, int cnx, int cny, const T* ec, T* et, int i0, int stride) {
  const T om = mg_omega2<T>();
  const int sx = L.fx - 1, sy = L.fy - 1, sz = L.fz - 1;           // the factors are 1 or 2
  auto vec = [&](int j, int x, int y, int z, T (&o)[VX]) {
    load_n<T, VX>(e + j, o);
    const T* row = ec + ((z >> sz) * cny + (y >> sy)) * cnx;
#pragma unroll
    for (int k = 0; k < VX; ++k) o[k] += row[(x + k) >> sx];
  };
  for (int i = i0; i < L.n / VX; i += stride) {
    const SubRow<T, VX> s(L, i);
    T uc[VX], fc[VX], res[VX];
    vec(s.c, s.x, s.y, s.z, uc);
    load_n<T, VX>(f + s.c, fc);
    sub_res<T, EPS, VX>(L, lo, hi, s, fc, uc, res, vec, [&](int j, int x, int y, int z) -> T {
      return e[j] + ec[((z >> sz) * cny + (y >> sy)) * cnx + (x >> sx)];
    });
#pragma unroll
    for (int k = 0; k < VX; ++k)
      uc[k] += om * sub_inv<T, EPS>(L, lo, hi, s.c + k, s.x + k, s.y, s.z) * res[k];
    store_n<T, VX>(et + s.c, uc);
  }
}

template <typename T, bool EPS, int VX>
__device__ __forceinline__ void sub_post2(const SubDesc<T>& L, const int8_t* lo, const int8_t* hi, const T* f,
                                          const T* et, T* e, int i0, int stride, Acc<T>& arz) {
  const T om = mg_omega1<T>();
  for (int i = i0; i < L.n / VX; i += stride) {
    const SubRow<T, VX> s(L, i);
    T vc[VX], fc[VX], res[VX];
    load_n<T, VX>(et + s.c, vc);
    load_n<T, VX>(f + s.c, fc);
    sub_res<T, EPS, VX>(
        L, lo, hi, s, fc, vc, res, [&](int j, int, int, int, T (&o)[VX]) { load_n<T, VX>(et + j, o); },
        [&](int j, int, int, int) -> T { return et[j]; });
#pragma unroll
    for (int k = 0; k < VX; ++k) {
      vc[k] += om * sub_inv<T, EPS>(L, lo, hi, s.c + k, s.x + k, s.y, s.z) * res[k];
      arz.add(fc[k], vc[k]);
    }
    arz.run();
    store_n<T, VX>(e + s.c, vc);
  }
}

// blob: the descriptors of the nl levels (SubDesc), then the face masks of
// those from solo on (nxy bytes each, lower face first): copied to shared
// memory in one pass of coalesced loads, as what the phases read first must
// not be fetched piecemeal (from the kernel parameters that took 3.3 us).
// solo: the first level that block 0 runs alone, its fields (and those of the
// levels below) in block 0's shared memory behind the blob.  last: level 0 of
// the launch is the finest one (z = e; r.z and beta go to the solver state);
// part: a double per block.
template <typename T, int NT, bool EPS>
__global__ void __launch_bounds__(NT, 1) k_mg_sub(const uint4* __restrict__ blob, int blob16, int nl, int solo,
                                               const double* __restrict__ cinv, int last, double* part, Scalars* S) {
  extern __shared__ __align__(16) unsigned char sub_smem[];
  __shared__ double fd[MG_MAX_COARSE];
  constexpr int V = 16 / sizeof(T);
  const int rank = blockIdx.x, nc = gridDim.x, tid = threadIdx.x;
  const int gt = rank * NT + tid, gs = nc * NT;
  for (int i = tid; i < blob16; i += NT) reinterpret_cast<uint4*>(sub_smem)[i] = blob[i];
  if (S->done) return;               // uniform over the cluster: nothing writes it before the last phase
  __syncthreads();
  const SubDesc<T>* const lv = reinterpret_cast<const SubDesc<T>*>(sub_smem);
  const int8_t* const masks = reinterpret_cast<const int8_t*>(sub_smem);
  T* const sm = reinterpret_cast<T*>(sub_smem);
  auto F = [&](int k) { return sm + lv[k].off; };
  auto E = [&](int k) { return sm + lv[k].off + lv[k].n; };
  auto ET = [&](int k) { return sm + lv[k].off + 2 * lv[k].n; };
  auto slo = [&](int k) { return masks + lv[k].moff; };
  auto shi = [&](int k) { return masks + lv[k].moff + lv[k].nxy; };
  const SubDesc<T>& B = lv[nl - 1];  // the coarsest level
  if (rank == 0 && B.n <= SUB_ROWS)  // its inverse: into the L1 by the time it is needed
    for (int i = tid; i * 16 < B.n * B.n; i += NT) asm volatile("prefetch.global.L1 [%0];" ::"l"(cinv + i * 16));
  Acc<T> arz, none;

  for (int k = 0; k < solo; ++k) {
    const SubDesc<T>&L = lv[k], &C = lv[k + 1];
    const bool vec = L.nx % V == 0 && L.n >= V * gs; // whole 16-byte vectors, enough for every thread
    if (k == 0) {
      if (vec) sub_pre<T, EPS, true, V>(L, L.tlo, L.thi, L.f, L.et, L.e, gt, gs);
      else sub_pre<T, EPS, true, 1>(L, L.tlo, L.thi, L.f, L.et, L.e, gt, gs);
    } else {
      if (vec) sub_pre<T, EPS, false, V>(L, L.tlo, L.thi, L.f, L.et, L.e, gt, gs);
      else sub_pre<T, EPS, false, 1>(L, L.tlo, L.thi, L.f, L.et, L.e, gt, gs);
    }
    cluster_sync();
    if (vec) sub_restrict<T, EPS, V>(L, L.tlo, L.thi, L.f, L.e, C, C.tlo, C.thi, C.f, C.et, gt, gs);
    else sub_restrict<T, EPS, 1>(L, L.tlo, L.thi, L.f, L.e, C, C.tlo, C.thi, C.f, C.et, gt, gs);
    cluster_sync();
  }
  if (rank == 0) {
    {
      const SubDesc<T>& L = lv[solo];
      T *fs = F(solo), *es = ET(solo);
      for (int c = tid; c < L.n; c += NT) {
        fs[c] = L.f[c];
        if (solo > 0) es[c] = L.et[c];
      }
      __syncthreads();
    }
    for (int k = solo; k + 1 < nl; ++k) {
      const SubDesc<T>& L = lv[k];
      if (k == 0) sub_pre<T, EPS, true, 1>(L, slo(k), shi(k), F(k), ET(k), E(k), tid, NT);
      else sub_pre<T, EPS, false, 1>(L, slo(k), shi(k), F(k), ET(k), E(k), tid, NT);
      __syncthreads();
      sub_restrict<T, EPS, 1>(L, slo(k), shi(k), F(k), E(k), lv[k + 1], slo(k + 1), shi(k + 1), F(k + 1), ET(k + 1), tid,
                           NT);
      __syncthreads();
    }
  }
  if (nc > 1 && B.n > SUB_ROWS) {                    // a row per warp over the cluster
    if (rank == 0 && solo < nl - 1) {
      const T* fs = F(nl - 1);
      for (int c = tid; c < B.n; c += NT) B.f[c] = fs[c];
    }
    cluster_sync();
    for (int c = tid; c < B.n; c += NT) fd[c] = (double)B.f[c];
    __syncthreads();
    const int lane = tid & 31;
    for (int row = gt >> 5; row < B.n; row += gs >> 5) {
      const double* a = cinv + (size_t)row * B.n;
      double acc = 0.0;
      for (int j = lane; j < B.n; j += 32) acc = fma(a[j], fd[j], acc);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
      if (lane == 0) B.e[row] = (T)acc;
    }
    cluster_sync();
    if (rank == 0) {
      T* es = E(nl - 1);
      for (int c = tid; c < B.n; c += NT) es[c] = B.e[c];
      __syncthreads();
    }
  } else if (rank == 0) {                            // a row per thread (the inverse is symmetric)
    const T* fs = F(nl - 1);
    for (int c = tid; c < B.n; c += NT) fd[c] = (double)fs[c];
    __syncthreads();
    for (int row = tid; row < B.n; row += NT) {
      double acc = 0.0;
      for (int j = 0; j < B.n; ++j) acc = fma(cinv[(size_t)j * B.n + row], fd[j], acc);
      E(nl - 1)[row] = (T)acc;
      if (solo == nl - 1) B.e[row] = (T)acc;
    }
    __syncthreads();
  }
  if (rank == 0) {
    for (int k = nl - 2; k >= solo; --k) {
      const SubDesc<T>&L = lv[k], &C = lv[k + 1];
      sub_post1<T, EPS, 1>(L, slo(k), shi(k), F(k), E(k), C.nx, C.ny, E(k + 1), ET(k), tid, NT);
      __syncthreads();
      sub_post2<T, EPS, 1>(L, slo(k), shi(k), F(k), ET(k), k == solo ? L.e : E(k), tid, NT, k == 0 ? arz : none);
      __syncthreads();
    }
  }
  for (int k = solo - 1; k >= 0; --k) {
    const SubDesc<T>&L = lv[k], &C = lv[k + 1];
    cluster_sync();                                  // the coarser level's e is complete
    const bool vec = L.nx % V == 0 && L.n >= V * gs;
    if (vec) sub_post1<T, EPS, V>(L, L.tlo, L.thi, L.f, L.e, C.nx, C.ny, C.e, L.et, gt, gs);
    else sub_post1<T, EPS, 1>(L, L.tlo, L.thi, L.f, L.e, C.nx, C.ny, C.e, L.et, gt, gs);
    cluster_sync();
    if (vec) sub_post2<T, EPS, V>(L, L.tlo, L.thi, L.f, L.et, L.e, gt, gs, k == 0 ? arz : none);
    else sub_post2<T, EPS, 1>(L, L.tlo, L.thi, L.f, L.et, L.e, gt, gs, k == 0 ? arz : none);
  }
  if (!last) return;
  typename SumOf<T>::type v[1] = {arz.sum()};
  const double d = block_sums<1, NT>(v, fd, tid);    // fd is free: NT pairs of floats or doubles
  if (tid == 0) part[rank] = d;
  cluster_sync();
  if (rank == 0 && tid == 0) {
    double rz = 0.0;
    for (int i = 0; i < nc; ++i) rz += __ldcg(part + i);
    if (!isfinite(rz)) {
      S->nonfinite = 1;
      S->status = 3;
      S->pending = 0;
      S->done = 1;
    } else {
      if (!S->first) S->beta = rz / S->rz;
      S->rz = rz;
    }
  }
}

// ----------------------------------------------------- the coarsest inverse

// The coarsest operator as a dense matrix, one row per thread; singular
// problems (no electrode) get shift added everywhere, which moves the zero
// eigenvalue of the constant vector to n shift.
template <typename T>
__global__ void __launch_bounds__(128) k_coarse_matrix(MgView<T> C, double shift, double* __restrict__ A) {
  const int n = (int)C.g.n, i = blockIdx.x * 128 + threadIdx.x;
  if (i >= n) return;
  for (int j = 0; j < n; ++j) A[(size_t)j * n + i] = shift;
  const int nx = C.g.nx, ny = C.g.ny, nz = C.g.nz, nxy = (int)C.g.nxy;
  const int x = i % nx, y = i / nx % ny, z = i / nxy;
  const double ec = C.eps ? (double)C.eps[i] : 1.0;
  double diag = 0.0;
  auto face = [&](int nb, double a) {
    const double en = C.eps ? (double)C.eps[nb] : 1.0;
    const double w = a * (2.0 * ec * en / (ec + en));
    diag += w;
    A[(size_t)nb * n + i] -= w;
  };
  face(i - x + (x == 0 ? nx - 1 : x - 1), (double)C.ax);
  face(i - x + (x == nx - 1 ? 0 : x + 1), (double)C.ax);
  face(i + ((y == 0 ? ny - 1 : y - 1) - y) * nx, (double)C.ay);
  face(i + ((y == ny - 1 ? 0 : y + 1) - y) * nx, (double)C.ay);
  const int xy = y * nx + x;
  if (z > 0) face(i - nxy, (double)C.az);
  else if (C.g.periodic_z) face(i + (nz - 1) * nxy, (double)C.az);
  else if (C.tlo[xy]) diag += 2.0 * ec * (double)C.az;
  if (z < nz - 1) face(i + nxy, (double)C.az);
  else if (C.g.periodic_z) face(i - (nz - 1) * nxy, (double)C.az);
  else if (C.thi[xy]) diag += 2.0 * ec * (double)C.az;
  A[(size_t)i * n + i] += diag;
}

// One Gauss-Jordan step (unknown k) at element (i, j) of a matrix whose
// columns are stored one after another.  With the unknowns before k done, the
// pivot row is the pivot column with the sign of the done entries turned.
__device__ __forceinline__ double gj_step(double a, int i, int j, int k, double ci, double cj, double p) {
  const double rj = (j < k ? -cj : cj) * p;
  if (i == k) return j == k ? p : rj;
  return j == k ? -ci * p : fma(-ci, rj, a);
}

// Step k over the whole matrix; col: the pivot column, next: the column of
// unknown k + 1 after the step.
constexpr int GJ_COLS = 8;
__global__ void __launch_bounds__(256) k_coarse_pivot(double* __restrict__ A, int n, int k,
                                                      const double* __restrict__ col, double* __restrict__ next) {
  const int i = blockIdx.x * 256 + threadIdx.x;
  __shared__ double p;
  if (threadIdx.x == 0) p = 1.0 / col[k];
  __syncthreads();
  if (i >= n) return;
  const double ci = col[i];
  for (int j = blockIdx.y * GJ_COLS; j < min(n, (int)(blockIdx.y + 1) * GJ_COLS); ++j) {
    const double v = gj_step(A[(size_t)j * n + i], i, j, k, ci, col[j], p);
    A[(size_t)j * n + i] = v;
    if (j == k + 1) next[i] = v;
  }
}

// All steps of a matrix of at most SUB_ROWS rows, in one block.
__global__ void __launch_bounds__(256) k_coarse_invert_small(double* __restrict__ A, int n) {
  __shared__ double a[SUB_ROWS * SUB_ROWS];
  __shared__ double col[SUB_ROWS];
  for (int e = threadIdx.x; e < n * n; e += 256) a[e] = A[e];
  __syncthreads();
  for (int k = 0; k < n; ++k) {
    if (threadIdx.x < n) col[threadIdx.x] = a[k * n + threadIdx.x];
    __syncthreads();
    const double p = 1.0 / col[k];
    for (int e = threadIdx.x; e < n * n; e += 256) {
      const int j = e / n, i = e - j * n;
      a[e] = gj_step(a[e], i, j, k, col[i], col[j], p);
    }
    __syncthreads();
  }
  for (int e = threadIdx.x; e < n * n; e += 256) A[e] = a[e];
}

// Singular problems: take the constant vector's eigenvalue out again, so that
// the product has zero mean whatever the mean of the right-hand side.
__global__ void __launch_bounds__(256) k_coarse_deflate(double* __restrict__ A, int n, double c) {
  for (size_t e = blockIdx.x * (size_t)256 + threadIdx.x; e < (size_t)n * n; e += (size_t)gridDim.x * 256) A[e] -= c;
}

// ---------------------------------------------------------------- launchers

template <typename T>
int launch_coarse_inverse(const LaunchCfg& L, const MgView<T>& C, int singular, double* cinv) {
  const int n = (int)C.g.n;
  const double shift = singular ? 2.0 * ((double)C.ax + (double)C.ay + (double)C.az) / n : 0.0;
  int launches = 2;
  k_coarse_matrix<T><<<(n + 127) / 128, 128, 0, L.stream>>>(C, shift, cinv);
  if (n <= SUB_ROWS) {
    k_coarse_invert_small<<<1, 256, 0, L.stream>>>(cinv, n);
  } else {
    double* const col = cinv + (size_t)n * n;        // two columns
    cudaMemcpyAsync(col, cinv, (size_t)n * sizeof(double), cudaMemcpyDeviceToDevice, L.stream);
    const dim3 grid((n + 255) / 256, (n + GJ_COLS - 1) / GJ_COLS);
    for (int k = 0; k < n; ++k)
      k_coarse_pivot<<<grid, 256, 0, L.stream>>>(cinv, n, k, col + (k & 1) * n, col + ((k + 1) & 1) * n);
    launches = 1 + n;
  }
  if (singular) {
    k_coarse_deflate<<<(int)std::min<size_t>(1024, ((size_t)n * n + 255) / 256), 256, 0, L.stream>>>(
        cinv, n, 1.0 / (shift * n * n));
    ++launches;
  }
  return launches;
}

template <typename T, bool EPS>
static cudaError_t mg_sub_t(const LaunchCfg& L, const MgTail& t, const void* blob, const double* cinv, int last,
                            double* part, Scalars* S) {
  constexpr int NT = SUB_THREADS;
  auto kernel = k_mg_sub<T, NT, EPS>;
  static int cluster = 0;                            // blocks per cluster that this device launches
  cudaLaunchConfig_t cfg{};
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.y = at.val.clusterDim.z = 1;
  cfg.blockDim = dim3(NT);
  cfg.stream = L.stream;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  if (cluster == 0) {
    allow_smem(kernel, MG_TAIL_SMEM);
    cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    cfg.dynamicSmemBytes = MG_TAIL_SMEM;
    int c = SUB_CLUSTER;
    for (; c > 1; c /= 2) {
      cfg.gridDim = dim3(c);
      at.val.clusterDim.x = c;
      int m = 0;
      if (cudaOccupancyMaxActiveClusters(&m, kernel, &cfg) == cudaSuccess && m > 0) break;
      cudaGetLastError();
    }
    cluster = c;
  }
  int nc = (t.solo > 0 || t.coarse > SUB_ROWS) ? cluster : 1;
  // FP32: no more blocks than its first level has 16-byte vectors for, but at
  // least 8.  A block holds its SM's registers while the first one runs the
  // solo levels: a batch of 30 films 17.15 ms with 16 blocks for every film,
  // 16.65 so (and 16.14 with 8 for every film, but then a film alone whose first
  // level has 65 536 cells pays 6 %).  FP64 levels are bound by the SMs' FP64
  // units: 8 blocks for 16 384 cells were 3 % slower.
  while (sizeof(T) == 4 && nc > 8 && t.cells <= (nc / 2) * NT * (int)(16 / sizeof(T))) nc /= 2;
  cfg.gridDim = dim3(nc);
  at.val.clusterDim.x = nc;
  cfg.dynamicSmemBytes = t.smem_bytes;
  return cudaLaunchKernelEx(&cfg, kernel, (const uint4*)blob, t.blob_bytes / 16, t.nl, t.solo, cinv, last, part, S);
}

template <typename T>
cudaError_t launch_mg_sub(const LaunchCfg& L, const MgTail& t, int eps, const void* blob, const double* cinv, int last,
                          double* part, Scalars* S) {
  return eps ? mg_sub_t<T, true>(L, t, blob, cinv, last, part, S) : mg_sub_t<T, false>(L, t, blob, cinv, last, part, S);
}

#define PF_COARSE_INSTANTIATE(T)                                                                           \
  template int launch_coarse_inverse<T>(const LaunchCfg&, const MgView<T>&, int, double*);                 \
  template cudaError_t launch_mg_sub<T>(const LaunchCfg&, const MgTail&, int, const void*, const double*, int,  \
                                        double*, Scalars*);

PF_COARSE_INSTANTIATE(float)
PF_COARSE_INSTANTIATE(double)

}  // namespace pf
