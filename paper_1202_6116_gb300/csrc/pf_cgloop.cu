// The whole Jacobi-PCG loop of a solve as one persistent launch (eps = 1).
//
// An iteration of k_cg_p and k_cg_r on a grid that fits in L2 spends most of
// its time between the kernels: on 32^3 (FP64) 24.7 us an iteration, of which
// the cells' FP64 arithmetic is 1.5 us, the rest launches, scalars passed
// through memory and two last-block reductions.  k_cg_loop keeps one block per
// SM resident for the whole solve (a cooperative launch): two barriers an
// iteration, after each of which every block sums the blocks' partials itself,
// in block order, so all hold the same alpha and beta and take the same
// decisions; one block writes the solver state at the end.  (Publishing the
// partials in slots that every block polls, without a counter, was 4 us an
// iteration slower: the polled lines are the written ones.  A 16-block cluster
// with its hardware barrier was 1 us faster on 32^3 and slower from 64 x 64 x
// 32 on.)
//
// A thread owns vectors of VX cells and walks its tile's planes with p of
// planes z - 1, z and z + 1 in registers; p at the in-plane neighbours is
// formed from r and p_old read through the L1 (no staging: the data are in
// L2, and nothing is left to overlap the copies with).
//
// Several films at once (a batch): the loop's blocks fill the GPU with few
// films, each waiting at its barriers.  Its work is split into virtual blocks, as
// many as a film alone has blocks, so that a film can run them in other ways with
// the same partials and the same order of the sums, that is the same bits: as the
// blocks of two ordinary launches an iteration (k_half_p, k_half_r), which the
// scheduler interleaves with the other films', or on fewer blocks of the loop, so
// that fewer films at a time keep their vectors in L2.  Which film does what:
// BatchLoops in pf_api.cu.
//
// The barrier's wait is bounded: a block that gives up marks the solve and
// leaves, and so do the others, each at its own limit.  The solve then ends as one
// that did not converge, and the call's later solves end before their first
// iteration (rhs_close), so that a call of many steps waits once.
#include <type_traits>

#include "pf_internal.h"
#include "pf_march.cuh"

namespace pf {

constexpr int LOOP_ROWS = 16;           // tile: 16 threads along x by 16 rows
// Largest vector the loop takes: its five then stay in L2.  (An iteration of
// 256 x 256 x 32 in FP32, 8 MB a vector, 24.8 us against 32.8 with two kernels;
// of 256 x 256 x 64, 16 MB, 45.7 against 42.4.  FP64, bound by its unit: 192 x 192
// x 48, 13.5 MB, 106.7 against 111.7; 256 x 256 x 32, 16 MB, 137.4 against 136.0.)
constexpr size_t LOOP_BYTES = 15u << 20;

// Sums of NV values over the block; value k in lane 0 of warp k.  FP32 pairs:
// a shuffle tree per warp, then one over the warps (a pair_add is 11 FP32
// operations; 32 of them in a row, as one warp over all threads would take,
// are 1400 cycles), each again in doubles where a pair leaves the range of a
// float.  scratch: 2 NV NT / 32 elements.  FP64: block_sums.
template <int NV, int NT>
__device__ __forceinline__ double loop_sums(const float2 (&v)[NV], void* scratch, int tid) {
  constexpr int NW = NT / 32;
  float2* sm = static_cast<float2*>(scratch);
  double* wide = reinterpret_cast<double*>(sm + NV * NW);
  const int lane = tid & 31, wid = tid >> 5;
#pragma unroll
  for (int k = 0; k < NV; ++k) {
    float2 d = v[k];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) d = pair_add(d, sum_xor(d, o));
    if (__any_sync(0xffffffffu, !isfinite(d.x))) {
      const double e = warp_total(sum_double(v[k]));
      if (lane == 0) wide[k * NW + wid] = e;
      d.x = NAN;
    }
    if (lane == 0) sm[k * NW + wid] = d;
  }
  __syncthreads();
  if (wid >= NV) return 0.0;
  const float2 w = lane < NW ? sm[wid * NW + lane] : make_float2(0.f, 0.f);
  float2 d = w;
#pragma unroll
  for (int o = NW / 2; o > 0; o >>= 1) d = pair_add(d, sum_xor(d, o));
  if (__any_sync(0xffffffffu, !isfinite(d.x))) return warp_total(isfinite(w.x) ? sum_double(w) : wide[wid * NW + lane]);
  return sum_double(d);
}
template <int NV, int NT>
__device__ __forceinline__ double loop_sums(const double (&v)[NV], void* scratch, int tid) {
  return block_sums<NV, NT>(v, scratch, tid);
}

// Virtual block vb's partials of NV values into set (nvb of each value).
template <int NV, int NT, typename V>
__device__ __forceinline__ void loop_partial(const V (&v)[NV], void* scratch, double* set, int vb, int nvb, int tid) {
  if (vb != (int)blockIdx.x) __syncthreads();          // the scratch may still be read
  const double d = loop_sums<NV, NT>(v, scratch, tid);
  if ((tid & 31) == 0 && (tid >> 5) < NV) set[(tid >> 5) * nvb + vb] = d;
}

// Sum of the nvb partials at v: the same in every warp that forms it.
__device__ __forceinline__ double loop_total(const double* v, int nvb, int lane) {
  double a = 0.0;
  for (int i = lane; i < nvb; i += 32) a += __ldcg(v + i);
  return warp_total(a);
}

// Sums of NV values over the nvb partials in set, in tot, after a barrier of
// all the grid's blocks: bar counts arrivals (zeroed by the right-hand side
// kernel), ph numbers the reductions.  The fence before the arrival orders the
// block's writes (it has met at a barrier since) before it.  The partials of
// reduction ph are rewritten at ph + 1 at the earliest, when every block has
// read them and arrived again: two sets in turn.  Returns false when the wait
// ran out.
template <int NV>
__device__ __forceinline__ bool loop_reduce(const double* set, unsigned* bar, int ph, int nvb, int tid, double* tot,
                                            int* ok, unsigned polls) {
  const int lane = tid & 31, wid = tid >> 5;
  __syncthreads();
  if (tid == 0) {
    __threadfence();
    atomicAdd(bar, 1u);
    const unsigned target = (unsigned)(ph + 1) * gridDim.x;      // (wraps with the count: compared as a difference)
    unsigned n = 0, c;
    do {
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(c) : "l"(bar) : "memory");
    } while ((int)(c - target) < 0 && ++n < polls);
    *ok = (int)(c - target) >= 0;
  }
  __syncthreads();
  if (!*ok) return false;
  if (wid < NV) {
    const double a = loop_total(set + wid * nvb, nvb, lane);
    if (lane == 0) tot[wid] = a;
  }
  __syncthreads();
  return true;
}

template <typename T>
struct LoopVecs {
  T *r, *p0, *p1, *q, *x;
};

// What an iteration knows when it begins.
template <typename T>
struct LoopIter {
  int first, pb, xz;       // first iteration; p_old is p1 (1) or p0; x is still 0
  T alpha, beta;           // of the last iteration
};

// First half of an iteration, over the block's virtual blocks: p = z + beta
// p_old, q = A p, x += alpha p_old; partials of p.q into set.
template <typename T, int VX, int G>
__device__ __forceinline__ void loop_p(const Geo& g, const Bc<T>& bc, const LoopVecs<T>& v, const LoopIter<T>& it,
                                       const MarchCfg& mc, int nvb, double* set, void* scratch, int tid) {
  constexpr int NT = 256 * G;
  using Sum = typename SumOf<T>::type;
  const int tx = threadIdx.x, nx = g.nx, ny = g.ny;
  const long long nxy = g.nxy;
  const T ih2 = T(g.ih2), inv6 = bc.itab[0], al = it.alpha, beta = it.beta;
  const bool first = it.first, xz = it.xz;
  const T* const r = v.r;
  const T* const pold = it.pb ? v.p1 : v.p0;
  T* const pnew = it.pb ? v.p0 : v.p1;
  auto zat = [&](T rv, int xy, int z) -> T { return rn_mul(rv, inv_diag_tab(g, bc, xy, z, inv6)); };
  // p at one cell, or at VX cells in a row, of plane z
  auto p1at = [&](long long zo, int xy, int z) -> T {
    const T zz = zat(r[zo + xy], xy, z);
    return first ? zz : rn_fma(beta, pold[zo + xy], zz);
  };
  auto pvec = [&](int xy, int z, T (&o)[VX], T (&old)[VX]) {
    const long long c = (long long)z * nxy + xy;
    T rv[VX];
    load_n<T, VX>(r + c, rv);
    if (!first) load_n<T, VX>(pold + c, old);
#pragma unroll
    for (int i = 0; i < VX; ++i) {
      const T zz = zat(rv[i], xy + i, z);
      o[i] = first ? zz : rn_fma(beta, old[i], zz);
    }
  };
  for (int vb = blockIdx.x; vb < nvb; vb += gridDim.x) {
    Acc<T> apq;
    for (long long t = vb * G + threadIdx.z; t < mc.ntiles; t += (long long)nvb * G) {
      const TileGeo<16, 16, VX> s = tile_geo<16, 16, VX>(g, t, mc);
      const bool lin = tx > 0, rin = tx < 15 && (tx + 1) * VX < s.w;
      const int ym = s.y == 0 ? ny - 1 : s.y - 1, yp = s.y == ny - 1 ? 0 : s.y + 1;
      const int xl = s.x == 0 ? nx - 1 : s.x - 1, xr = s.x + VX >= nx ? 0 : s.x + VX;
      T pm[VX], pc[VX], pp[VX], oc[VX], op[VX], t0[VX];
#pragma unroll
      for (int i = 0; i < VX; ++i) pm[i] = pc[i] = pp[i] = oc[i] = op[i] = t0[i] = T(0);
      if (s.act) {
        const int zb = z_below(g, s.z0);
        if (zb >= 0) pvec(s.xy, zb, pm, t0);
        pvec(s.xy, s.z0, pc, oc);
      }
      for (int z = s.z0; z < s.z1; ++z) {
        const int zb = z_below(g, z), za = z_above(g, z);
        const long long zo = (long long)z * nxy;
        T pym[VX], pyp[VX], xv[VX];
        T pl = __shfl_up_sync(0xffffffffu, pc[VX - 1], 1), pr = __shfl_down_sync(0xffffffffu, pc[0], 1);
        if (s.act) {
          if (za >= 0) pvec(s.xy, za, pp, op);
          pvec(ym * nx + s.x, z, pym, t0);
          pvec(yp * nx + s.x, z, pyp, t0);
          if (!lin) pl = p1at(zo, s.y * nx + xl, z);
          if (!rin) pr = p1at(zo, s.y * nx + xr, z);
          if (!first && !xz) load_n<T, VX>(v.x + zo + s.xy, xv);
          T qv[VX];
          const bool bt = zb < 0 || za < 0;
#pragma unroll
          for (int i = 0; i < VX; ++i) {
            Stencil7<T> st;
            st.c = pc[i];
            st.xm = i == 0 ? pl : pc[i - 1];
            st.xp = i == VX - 1 ? pr : pc[i + 1];
            st.ym = pym[i];
            st.yp = pyp[i];
            st.zm = pm[i];
            st.zp = pp[i];
            st.zb = zb;
            st.za = za;
            const int dlo = (bt && zb < 0) ? (int)bc.tlo[s.xy + i] : 0;
            const int dhi = (bt && za < 0) ? (int)bc.thi[s.xy + i] : 0;
            qv[i] = apply_bt(st, dlo, dhi, ih2, bt);
            apq.add(pc[i], qv[i]);
            if (!first) xv[i] = xz ? rn_mul(al, oc[i]) : rn_fma(al, oc[i], xv[i]);
          }
          apq.run();
          if (!first) store_n<T, VX>(v.x + zo + s.xy, xv);
          store_n<T, VX>(pnew + zo + s.xy, pc);
          store_n<T, VX>(v.q + zo + s.xy, qv);
        }
#pragma unroll
        for (int i = 0; i < VX; ++i) {
          pm[i] = pc[i];
          pc[i] = pp[i];
          oc[i] = op[i];
        }
      }
    }
    const Sum sum[1] = {apq.sum()};
    loop_partial<1, NT>(sum, scratch, set, vb, nvb, tid);
  }
}

// Second half: r -= alpha q over the same tiles; partials of r.r and r.z.
template <typename T, int VX, int G>
__device__ __forceinline__ void loop_r(const Geo& g, const Bc<T>& bc, const LoopVecs<T>& v, T alpha, const MarchCfg& mc,
                                       int nvb, double* set, void* scratch, int tid) {
  constexpr int NT = 256 * G;
  using Sum = typename SumOf<T>::type;
  const T inv6 = bc.itab[0];
  for (int vb = blockIdx.x; vb < nvb; vb += gridDim.x) {
    Acc<T> arr, arz;
    for (long long t = vb * G + threadIdx.z; t < mc.ntiles; t += (long long)nvb * G) {
      const TileGeo<16, 16, VX> s = tile_geo<16, 16, VX>(g, t, mc);
      if (!s.act) continue;
      for (int z = s.z0; z < s.z1; ++z) {
        const long long c = (long long)z * g.nxy + s.xy;
        T rv[VX], qv[VX];
        load_n<T, VX>(v.r + c, rv);
        load_n<T, VX>(v.q + c, qv);
#pragma unroll
        for (int i = 0; i < VX; ++i) {
          rv[i] = rn_fma(-alpha, qv[i], rv[i]);
          arr.add(rv[i], rv[i]);
          arz.add(rv[i], rn_mul(rv[i], inv_diag_tab(g, bc, s.xy + i, z, inv6)));
        }
        arr.run();
        arz.run();
        store_n<T, VX>(v.r + c, rv);
      }
    }
    const Sum sum[2] = {arr.sum(), arz.sum()};
    loop_partial<2, NT>(sum, scratch, set, vb, nvb, tid);
  }
}

template <typename T, int VX, int G>
__global__ void __launch_bounds__(256 * G)
k_cg_loop(Geo g, Bc<T> bc, LoopVecs<T> v, double* part, Scalars* S, MarchCfg mc, int nvb, unsigned polls) {
  constexpr int NT = 256 * G;
  __shared__ typename SumOf<T>::type scratch[2 * NT];
  __shared__ double tot[2], alpha_s, beta_s, rel_s;
  __shared__ int verdict, ok;           // verdict: 0 go on, 1 converged, 2 maxit, 3 breakdown, 4 non-finite
  if (S->done) return;                  // written by this kernel only after the last barrier
  const int tid = threadIdx.x + 16 * threadIdx.y + 256 * threadIdx.z;
  const double rtol = S->rtol, bnorm = S->bnorm;
  const int maxit = S->maxit;
  double rz = S->rz, rr = 0.0, rel = S->last_rel, alpha = 0.0;
  LoopIter<T> it{1, S->pbuf, S->xzero, T(0), T(0)};
  int iter = 0, ph = 0;

  for (;;) {
    double* set = part + (size_t)(ph & 1) * 2 * nvb;
    loop_p<T, VX, G>(g, bc, v, it, mc, nvb, set, scratch, tid);
    // alpha = r.z / p.q
    {
      if (!loop_reduce<1>(set, &S->bar, ph++, nvb, tid, tot, &ok, polls)) {
        if (tid == 0) S->timeout = S->status = 3;
        return;
      }
      if (tid == 0) {
        const double a = tot[0];
        verdict = (a > 0.0) ? 0 : (isfinite(a) ? 3 : 4);
        alpha_s = (a > 0.0) ? rz / a : 0.0;
      }
      __syncthreads();
    }
    if (!it.first) it.xz = 0;
    ++iter;
    it.first = 0;
    it.pb ^= 1;
    alpha = alpha_s;
    if (verdict) break;                 // breakdown: stop with the current iterate
    it.alpha = T(alpha);
    set = part + (size_t)(ph & 1) * 2 * nvb;
    loop_r<T, VX, G>(g, bc, v, it.alpha, mc, nvb, set, scratch, tid);
    {
      if (!loop_reduce<2>(set, &S->bar, ph++, nvb, tid, tot, &ok, polls)) {
        if (tid == 0) S->timeout = S->status = 3;
        return;
      }
      if (tid == 0) {
        rel_s = sqrt(tot[0]) / bnorm;
        verdict = !isfinite(tot[0]) ? 4 : rel_s < rtol ? 1 : iter >= maxit ? 2 : 0;
      }
      if (tid == 32) beta_s = tot[1] / rz;
      __syncthreads();
      rel = rel_s;
      rr = tot[0];
    }
    if (verdict) break;
    it.beta = T(beta_s);
    rz = tot[1];
  }
  if (blockIdx.x != 0 || tid != 0) return;
  S->iter = iter;
  S->pbuf = it.pb;
  S->first = 0;
  S->xzero = it.xz;
  S->alpha = alpha;
  S->rz = rz;
  if (verdict == 1 || verdict == 2 || verdict == 4) {
    S->rr = rr;
    S->last_rel = rel;
  }
  S->pending = verdict == 1 || verdict == 2;
  if (verdict != 1) S->status = 3;
  if (verdict == 4) S->nonfinite = 1;
  S->done = 1;
}

// The two halves of an iteration as launches of their own, a virtual block per
// block: the same partials in the same order, so the same bits as the loop.  (64
// films of 64 x 64 x 32 in FP32: 59 us an iteration for all of them, 302 MB through
// L2; two plane marches 66 us.)
template <typename T, int VX, int G>
__global__ void __launch_bounds__(256 * G)
k_half_p(Geo g, Bc<T> bc, LoopVecs<T> v, double* part, Scalars* S, MarchCfg mc) {
  constexpr int NT = 256 * G;
  __shared__ typename SumOf<T>::type scratch[2 * NT];
  if (S->done) return;
  const int tid = threadIdx.x + 16 * threadIdx.y + 256 * threadIdx.z, nvb = gridDim.x;
  const LoopIter<T> it{S->first, S->pbuf, S->xzero, T(S->alpha), T(S->beta)};
  loop_p<T, VX, G>(g, bc, v, it, mc, nvb, part, scratch, tid);
  if (!last_block<NT>(&S->ticket) || tid >= 32) return;
  const double a = loop_total(part, nvb, tid);
  if (tid != 0) return;
  S->iter += 1;
  S->pbuf = it.pb ^ 1;
  if (!it.first) S->xzero = 0;
  S->first = 0;
  S->alpha = (a > 0.0) ? S->rz / a : 0.0;
  if (!(a > 0.0)) {                     // breakdown (or NaN): stop with the current iterate
    if (!isfinite(a)) S->nonfinite = 1;
    S->pending = 0;
    S->status = 3;
    S->done = 1;
  }
  S->ticket = 0;
}

template <typename T, int VX, int G>
__global__ void __launch_bounds__(256 * G)
k_half_r(Geo g, Bc<T> bc, LoopVecs<T> v, double* part, Scalars* S, MarchCfg mc, cudaGraphConditionalHandle cond) {
  constexpr int NT = 256 * G;
  __shared__ typename SumOf<T>::type scratch[2 * NT];
  const int tid = threadIdx.x + 16 * threadIdx.y + 256 * threadIdx.z, nvb = gridDim.x;
  if (S->done) {                        // a breakdown in k_half_p ends the loop
    if (blockIdx.x == 0 && tid == 0) cudaGraphSetConditional(cond, 0u);
    return;
  }
  loop_r<T, VX, G>(g, bc, v, T(S->alpha), mc, nvb, part, scratch, tid);
  if (!last_block<NT>(&S->ticket) || tid >= 32) return;
  const double rr = loop_total(part, nvb, tid), rz = loop_total(part + nvb, nvb, tid);
  if (tid != 0) return;
  const double rel = sqrt(rr) / S->bnorm;
  S->rr = rr;
  S->last_rel = rel;
  if (!isfinite(rr)) {
    S->nonfinite = 1;
    S->status = 3;
    S->pending = 0;
    S->done = 1;
  } else if (rel < S->rtol) {
    S->pending = 1;
    S->done = 1;
  } else if (S->iter >= S->maxit) {
    S->pending = 1;
    S->status = 3;
    S->done = 1;
  } else {
    S->beta = rz / S->rz;
    S->rz = rz;
  }
  S->ticket = 0;
  cudaGraphSetConditional(cond, S->done ? 0u : 1u);
}

// ---------------------------------------------------------------- launchers

// Tiles for streams groups of threads, each walking tiles one after another:
// the depth of least rounds x (planes + 2) (a tile starts with two loads of
// its own column).
static MarchCfg loop_tiles(const Geo& g, int vx, long long streams) {
  MarchCfg m{};
  m.vx = vx;
  m.tiles_x = (g.nx + 16 * vx - 1) / (16 * vx);
  m.tiles_y = (g.ny + LOOP_ROWS - 1) / LOOP_ROWS;
  const long long cols = (long long)m.tiles_x * m.tiles_y;
  long long best = 0;
  for (int tz = 1; tz <= g.nz; ++tz) {
    const long long tiles = cols * ((g.nz + tz - 1) / tz), cost = (tiles + streams - 1) / streams * (tz + 2);
    if (best == 0 || cost <= best) {
      best = cost;
      m.tz = tz;
      m.ntiles = tiles;
    }
  }
  return m;
}

// Virtual blocks and tiles of a film's loop.
static int loop_blocks(const LaunchCfg& L, const Geo& g, int vx, int groups, MarchCfg& mc) {
  mc = loop_tiles(g, vx, (long long)L.nsm * groups);
  return (int)std::min<long long>(L.nsm, (mc.ntiles + groups - 1) / groups);
}

// Blocks of the loop that an SM holds at a time; 0: it cannot be launched here.
template <typename T, int VX, int G>
static int loop_resident() {
  static int n = -1;
  if (n < 0) {
    int nb = 0, coop = 0, dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_cg_loop<T, VX, G>, 256 * G, 0) != cudaSuccess)
      coop = 0;
    cudaGetLastError();
    n = coop ? nb : 0;
  }
  return n;
}

// dry: only whether it can be launched here.
template <typename T, int VX, int G>
static bool cg_loop_t(const LaunchCfg& L, const Geo& g, const Dev<T>& d, bool dry) {
  auto kernel = k_cg_loop<T, VX, G>;
  const bool can = loop_resident<T, VX, G>() > 0;
  if (dry || !can) return can;
  MarchCfg mc;
  const int nvb = loop_blocks(L, g, VX, G, mc);
  cudaLaunchConfig_t cfg{};
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeCooperative;
  at.val.cooperative = 1;
  cfg.gridDim = dim3((unsigned)((nvb + L.loop_share - 1) / L.loop_share));
  cfg.blockDim = dim3(16, 16, G);
  cfg.stream = L.stream;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  const LoopVecs<T> v{d.r, d.p0, d.p1, d.q, d.phi};
  return cudaLaunchKernelEx(&cfg, kernel, g, d.bc, v, d.part, d.S, mc, nvb, L.loop_polls) == cudaSuccess;
}

template <typename T, int VX, int G>
static void cg_halves_t(const LaunchCfg& L, const Geo& g, const Dev<T>& d, cudaGraphConditionalHandle cond) {
  MarchCfg mc;
  const int nvb = loop_blocks(L, g, VX, G, mc);
  const dim3 block(16, 16, G);
  const LoopVecs<T> v{d.r, d.p0, d.p1, d.q, d.phi};
  k_half_p<T, VX, G><<<nvb, block, 0, L.stream>>>(g, d.bc, v, d.part, d.S, mc);
  k_half_r<T, VX, G><<<nvb, block, 0, L.stream>>>(g, d.bc, v, d.part, d.S, mc, cond);
}

// Calls f with the cells of a film's threads and the thread groups of its blocks.
// Films that do not fill the GPU take vectors all the same (half as long where 16 of
// them are longer than a row) and one group a block: ms a step of a film alone 0.123
// on 32^3 and 0.127 on 64 x 64 x 32 in FP32, where single cells and four groups took
// 0.136 and 0.143, and 0.169 against 0.177 on 32^3 in FP64 (vectors with two groups:
// 0.206); 64 such films as two launches an iteration 1.87, 3.9 and 3.35, where single
// cells took 2.47, 8.4 and 4.6 and two plane marches take 2.15, 4.34 and 3.78.  Rows of
// no whole vectors (101 x 75 x 19) keep four groups in FP32, 0.191 against 0.223.
template <typename T, class F>
static auto loop_form(const LaunchCfg& L, const Geo& g, F f) {
  constexpr int V = 16 / sizeof(T), F32 = sizeof(T) == 4;
  const bool vec = L.march.vx == V;
  using std::integral_constant;
  if (loop_fills(L, g)) {
    if (vec) return f(integral_constant<int, V>(), integral_constant<int, 2>());
    return f(integral_constant<int, 1>(), integral_constant<int, F32 ? 4 : 2>());
  }
  if (vec && 16 * (V / 2) >= g.nx) return f(integral_constant<int, V / 2>(), integral_constant<int, 1>());
  if (vec) return f(integral_constant<int, V>(), integral_constant<int, 1>());
  return f(integral_constant<int, 1>(), integral_constant<int, F32 ? 4 : 1>());
}

template <typename T>
bool launch_cg_loop(const LaunchCfg& L, const Geo& g, const Dev<T>& d, bool dry) {
  if (d.eps || (size_t)g.n * sizeof(T) > LOOP_BYTES) return false;
  return loop_form<T>(L, g, [&](auto vx, auto groups) { return cg_loop_t<T, vx, groups>(L, g, d, dry); });
}

template <typename T>
int cg_loop_blocks(const LaunchCfg& L, const Geo& g, int* held) {
  MarchCfg mc;
  return loop_form<T>(L, g, [&](auto vx, auto groups) {
    *held = loop_resident<T, vx, groups>() * L.nsm;
    return loop_blocks(L, g, vx, groups, mc);
  });
}

template <typename T>
void launch_cg_halves(const LaunchCfg& L, const Geo& g, const Dev<T>& d, cudaGraphConditionalHandle cond) {
  loop_form<T>(L, g, [&](auto vx, auto groups) { cg_halves_t<T, vx, groups>(L, g, d, cond); });
}

#define PF_LOOP_INSTANTIATE(T)                                                              \
  template bool launch_cg_loop<T>(const LaunchCfg&, const Geo&, const Dev<T>&, bool);       \
  template int cg_loop_blocks<T>(const LaunchCfg&, const Geo&, int*);                       \
  template void launch_cg_halves<T>(const LaunchCfg&, const Geo&, const Dev<T>&, cudaGraphConditionalHandle);

PF_LOOP_INSTANTIATE(float)
PF_LOOP_INSTANTIATE(double)

}  // namespace pf
