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
// films, each waiting at its barriers, where two kernels an iteration had
// interleaved all (64 films of 32^3 in FP32: 3.36 ms a step against 2.07).  The
// work is therefore split into virtual blocks, as many as a film alone has
// blocks, and a film in a batch runs them on an eighth of the blocks: same
// partials, same order of the sums, same bits, more films side by side.
//
// The barrier's wait is bounded: a block that gives up marks the solve and
// leaves, and so do the others, each at its own limit.
#include "pf_internal.h"
#include "pf_march.cuh"

namespace pf {

constexpr int LOOP_ROWS = 16;           // tile: 16 threads along x by 16 rows
// Largest vector the loop takes: its five then stay in L2.  (An iteration of
// 256 x 256 x 32 in FP32, 8 MB a vector, 24.8 us against 32.8 with two kernels;
// of 256 x 256 x 64, 16 MB, 45.7 against 42.4.  FP64, bound by its unit: 192 x 192
// x 48, 13.5 MB, 106.7 against 111.7; 256 x 256 x 32, 16 MB, 137.4 against 136.0.)
constexpr size_t LOOP_BYTES = 15u << 20;
constexpr unsigned LOOP_SPIN = 1u << 22;   // polls before a barrier gives up (seconds)

template <typename T, int VX>
struct LoopGroups {                     // tiles a block walks at once (registers: 64 or 128 a thread)
  static constexpr int value = sizeof(T) * VX <= 4 ? 4 : 2;
};

// Sums of NV values over the block; value k in lane 0 of warp k.  FP32 pairs:
// a shuffle tree per warp, then one over the warps (a pair_add is 11 FP32
// operations; 32 of them in a row, as one warp over all threads would take,
// are 1400 cycles).  FP64: block_sums.
template <int NV, int NT>
__device__ __forceinline__ double loop_sums(const float2 (&v)[NV], void* scratch, int tid) {
  float2* sm = static_cast<float2*>(scratch);
  constexpr int NW = NT / 32;
  const int lane = tid & 31, wid = tid >> 5;
#pragma unroll
  for (int k = 0; k < NV; ++k) {
    float2 d = v[k];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) d = pair_add(d, sum_xor(d, o));
    if (lane == 0) sm[k * NW + wid] = d;
  }
  __syncthreads();
  if (wid >= NV) return 0.0;
  float2 d = lane < NW ? sm[wid * NW + lane] : make_float2(0.f, 0.f);
#pragma unroll
  for (int o = NW / 2; o > 0; o >>= 1) d = pair_add(d, sum_xor(d, o));
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

// Sums of NV values over the nvb partials in set, in tot, after a barrier of
// all the grid's blocks: bar counts arrivals (zeroed by the right-hand side
// kernel), ph numbers the reductions.  The fence before the arrival orders the
// block's writes (it has met at a barrier since) before it.  The partials of
// reduction ph are rewritten at ph + 1 at the earliest, when every block has
// read them and arrived again: two sets in turn.  Returns false when the wait
// ran out.
template <int NV>
__device__ __forceinline__ bool loop_reduce(const double* set, unsigned* bar, int ph, int nvb, int tid, double* tot,
                                            int* ok) {
  const int lane = tid & 31, wid = tid >> 5;
  __syncthreads();
  if (tid == 0) {
    __threadfence();
    atomicAdd(bar, 1u);
    const unsigned target = (unsigned)(ph + 1) * gridDim.x;      // (wraps with the count: compared as a difference)
    unsigned n = 0, c;
    do {
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(c) : "l"(bar) : "memory");
    } while ((int)(c - target) < 0 && ++n < LOOP_SPIN);
    *ok = (int)(c - target) >= 0;
  }
  __syncthreads();
  if (!*ok) return false;
  if (wid < NV) {
    double a = 0.0;
    for (int i = lane; i < nvb; i += 32) a += __ldcg(set + wid * nvb + i);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
    if (lane == 0) tot[wid] = a;
  }
  __syncthreads();
  return true;
}

template <typename T, int VX>
__global__ void __launch_bounds__(256 * LoopGroups<T, VX>::value)
k_cg_loop(Geo g, Bc<T> bc, T* r, T* p0, T* p1, T* q, T* x, double* part, Scalars* S, MarchCfg mc, int nvb) {
  constexpr int G = LoopGroups<T, VX>::value, NT = 256 * G;
  using Sum = typename SumOf<T>::type;
  __shared__ Sum scratch[2 * NT];
  __shared__ double tot[2], alpha_s, beta_s, rel_s;
  __shared__ int verdict, ok;           // verdict: 0 go on, 1 converged, 2 maxit, 3 breakdown, 4 non-finite
  if (S->done) return;                  // written by this kernel only after the last barrier
  const int tx = threadIdx.x, ty = threadIdx.y, tid = tx + 16 * ty + 256 * threadIdx.z;
  const int nx = g.nx, ny = g.ny;
  const long long nxy = g.nxy;
  const T ih2 = T(g.ih2);
  const T inv6 = bc.itab[0];
  auto inv_at = [&](int xy, int z) -> T { return inv_diag_tab(g, bc, xy, z, inv6); };
  const double rtol = S->rtol, bnorm = S->bnorm;
  const int maxit = S->maxit;
  double rz = S->rz, rr = 0.0, rel = S->last_rel, alpha = 0.0;
  T beta = T(0);
  int pb = S->pbuf, iter = 0, xz = S->xzero;
  int ph = 0;

  for (;;) {
    const bool first = iter == 0;
    const T* const pold = pb ? p1 : p0;
    T* const pnew = pb ? p0 : p1;
    const T al = T(alpha);
    // p at one cell, or at VX cells in a row, of plane z
    auto p1at = [&](long long zo, int xy, int z) -> T {
      const T zz = r[zo + xy] * inv_at(xy, z);
      return first ? zz : zz + beta * pold[zo + xy];
    };
    auto pvec = [&](int xy, int z, T (&o)[VX], T (&old)[VX]) {
      const long long c = (long long)z * nxy + xy;
      T rv[VX];
      load_n<T, VX>(r + c, rv);
      if (!first) load_n<T, VX>(pold + c, old);
#pragma unroll
      for (int i = 0; i < VX; ++i) {
        const T zz = rv[i] * inv_at(xy + i, z);
        o[i] = first ? zz : zz + beta * old[i];
      }
    };
    double* set = part + (size_t)(ph & 1) * 2 * nvb;
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
            if (!first && !xz) load_n<T, VX>(x + zo + s.xy, xv);
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
              if (!first) xv[i] = xz ? al * oc[i] : xv[i] + al * oc[i];
            }
            apq.run();
            if (!first) store_n<T, VX>(x + zo + s.xy, xv);
            store_n<T, VX>(pnew + zo + s.xy, pc);
            store_n<T, VX>(q + zo + s.xy, qv);
          }
#pragma unroll
          for (int i = 0; i < VX; ++i) {
            pm[i] = pc[i];
            pc[i] = pp[i];
            oc[i] = op[i];
          }
        }
      }
      const Sum v[1] = {apq.sum()};
      loop_partial<1, NT>(v, scratch, set, vb, nvb, tid);
    }
    // alpha = r.z / p.q
    {
      if (!loop_reduce<1>(set, &S->bar, ph++, nvb, tid, tot, &ok)) {
        if (tid == 0) S->timeout = 1;
        return;
      }
      if (tid == 0) {
        const double a = tot[0];
        verdict = (a > 0.0) ? 0 : (isfinite(a) ? 3 : 4);
        alpha_s = (a > 0.0) ? rz / a : 0.0;
      }
      __syncthreads();
    }
    if (!first) xz = 0;
    ++iter;
    pb ^= 1;
    alpha = alpha_s;
    if (verdict) break;                 // breakdown: stop with the current iterate
    // r -= alpha q over the same tiles, r.r and r.z
    const T aq = T(alpha);
    set = part + (size_t)(ph & 1) * 2 * nvb;
    for (int vb = blockIdx.x; vb < nvb; vb += gridDim.x) {
      Acc<T> arr, arz;
      for (long long t = vb * G + threadIdx.z; t < mc.ntiles; t += (long long)nvb * G) {
        const TileGeo<16, 16, VX> s = tile_geo<16, 16, VX>(g, t, mc);
        if (!s.act) continue;
        for (int z = s.z0; z < s.z1; ++z) {
          const long long c = (long long)z * nxy + s.xy;
          T rv[VX], qv[VX];
          load_n<T, VX>(r + c, rv);
          load_n<T, VX>(q + c, qv);
#pragma unroll
          for (int i = 0; i < VX; ++i) {
            rv[i] = rv[i] - aq * qv[i];
            arr.add(rv[i], rv[i]);
            arz.add(rv[i], rv[i] * inv_at(s.xy + i, z));
          }
          arr.run();
          arz.run();
          store_n<T, VX>(r + c, rv);
        }
      }
      const Sum v[2] = {arr.sum(), arz.sum()};
      loop_partial<2, NT>(v, scratch, set, vb, nvb, tid);
    }
    {
      if (!loop_reduce<2>(set, &S->bar, ph++, nvb, tid, tot, &ok)) {
        if (tid == 0) S->timeout = 1;
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
    beta = T(beta_s);
    rz = tot[1];
  }
  if (blockIdx.x != 0 || tid != 0) return;
  S->iter = iter;
  S->pbuf = pb;
  S->first = 0;
  S->xzero = xz;
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

// dry: only whether it can be launched here.
template <typename T, int VX>
static bool cg_loop_t(const LaunchCfg& L, const Geo& g, const Dev<T>& d, bool dry) {
  constexpr int G = LoopGroups<T, VX>::value;
  auto kernel = k_cg_loop<T, VX>;
  static int blocks = -1;               // blocks of the grid (0: cannot be launched here)
  if (blocks < 0) {
    int nb = 0, coop = 0, dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, kernel, 256 * G, 0) != cudaSuccess)
      coop = 0;
    cudaGetLastError();
    blocks = coop && nb > 0 ? L.nsm : 0;
  }
  if (dry || blocks == 0) return blocks > 0;
  const MarchCfg mc = loop_tiles(g, VX, (long long)blocks * G);
  cudaLaunchConfig_t cfg{};
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeCooperative;
  at.val.cooperative = 1;
  const int nvb = (int)std::min<long long>(blocks, (mc.ntiles + G - 1) / G);
  cfg.gridDim = dim3((unsigned)((nvb + L.loop_share - 1) / L.loop_share));
  cfg.blockDim = dim3(16, 16, G);
  cfg.stream = L.stream;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, g, d.bc, d.r, d.p0, d.p1, d.q, d.phi, d.part, d.S, mc, nvb) == cudaSuccess;
}

template <typename T>
bool launch_cg_loop(const LaunchCfg& L, const Geo& g, const Dev<T>& d, bool dry) {
  constexpr int V = 16 / sizeof(T);
  if (d.eps || (size_t)g.n * sizeof(T) > LOOP_BYTES) return false;
  // vectors when they are enough to occupy every thread
  const bool vec = L.march.vx == V && g.n / V >= (long long)L.nsm * 256 * LoopGroups<T, V>::value;
  return vec ? cg_loop_t<T, V>(L, g, d, dry) : cg_loop_t<T, 1>(L, g, d, dry);
}

template bool launch_cg_loop<float>(const LaunchCfg&, const Geo&, const Dev<float>&, bool);
template bool launch_cg_loop<double>(const LaunchCfg&, const Geo&, const Dev<double>&, bool);

}  // namespace pf
