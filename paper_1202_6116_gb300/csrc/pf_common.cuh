// Internal device helpers of the GPU library: grid geometry, boundary masks,
// FP64-accurate reductions and the solver scalar block.  Not part of the ABI.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <type_traits>

namespace pf {

// Tile of one thread block in the simple per-cell kernels: TX x TY columns of
// tz cells (x fastest).
constexpr int TX = 32;
constexpr int TY = 8;
constexpr int NTHREADS = TX * TY;
// Threads of a plane-march block (MTX x MTY, each owning one 16-byte vector
// of cells in x) and block size of the flat kernels.
constexpr int MTX = 16;
constexpr int MTY = 16;
constexpr int FLAT_THREADS = 256;

// Tiling of a plane-march launch: tiles of (MTX * vx) x MTY columns times tz
// planes; vx = cells per thread (16 bytes, or 1 when nx is not a multiple).
// Tile z-index iz covers planes [zlo + iz (tz + zskip), that + tz), clipped
// at nz - zcut; all three are 0 for a launch over the whole z range (a launch
// over the interior planes sets zlo = zcut = b; one over the two face slabs
// of b planes sets tz = b, zskip = nz - 2 b).
struct MarchCfg {
  int tiles_x, tiles_y, tz;
  long long ntiles;
  int grid;
  int vx;
  int zlo, zcut, zskip;
  int bps;           // resident blocks per SM asked for (0: as many as fit; kernels
                     // with their own occupancy size their grid by it)
};

struct Geo {
  int nx, ny, nz;
  int periodic_z;
  int zair;                // first air plane (nz: no air layers); P = 0 from there up
  long long nxy, n;
  double ih, ih2;          // 1/dx, 1/dx^2
  int tz;                  // cells per column in one tile
  int tiles_x, tiles_y, tiles_z;
  long long ntiles;
};

// Electrical z-face masks (per (x,y) cell of the face).
template <typename T>
struct Bc {
  const int8_t* tlo;
  const int8_t* thi;
  const T* vlo;
  const T* vhi;
  T itab[9];               // 1/diag(A) with eps = 1, by 3 (kind of the lower z face) + kind of the upper one
                           // (0 interior, 1 open, 2 electrode); see diag_table
};

// faces_of: the weight of a z face of each kind in the diagonal.  The nine
// values are formed on the host: a division is 20 FP64 operations, and one per
// thread at the start of a kernel is 6 us on an SM's FP64 unit.
inline int faces_of(int kind) { return kind == 0 ? 1 : 2 * (kind - 1); }
template <typename T>
inline void diag_table(double ih2, T (&tab)[9]) {
  for (int i = 0; i < 9; ++i) tab[i] = T(1) / (T(4 + faces_of(i / 3) + faces_of(i % 3)) * T(ih2));
}

// 16-byte vector type of a field element type.
template <typename T>
struct Vec16;
template <>
struct Vec16<float> {
  using type = float4;
};
template <>
struct Vec16<double> {
  using type = double2;
};

// 1/diag(A) at column xy of plane z when eps = 1.  The diagonal is
// (interior faces + 2 x electrode faces)/dx^2: 6/dx^2 away from the z faces.
// The table holds the same bits as the division, so z = r/diag agrees bit for
// bit between kernels whichever of these they use.
template <typename T>
__device__ __forceinline__ T inv_diag_tab(const Geo& g, const Bc<T>& bc, long long xy, int z, T inv6) {
  if (g.periodic_z || (z > 0 && z < g.nz - 1)) return inv6;
  return bc.itab[3 * (z > 0 ? 0 : 1 + (int)bc.tlo[xy]) + (z < g.nz - 1 ? 0 : 1 + (int)bc.thi[xy])];
}
// The plane-march and flat kernels divide in FP32: indexing the kernel
// parameters there slowed the Jacobi iteration of a 256 x 256 x 64 film from
// 41.0 to 44.7 us.
template <typename T>
__device__ __forceinline__ T inv_diag_unit(const Geo& g, const Bc<T>& bc, long long xy, int z, T inv6) {
  if constexpr (sizeof(T) == 8) return inv_diag_tab(g, bc, xy, z, inv6);
  if (g.periodic_z || (z > 0 && z < g.nz - 1)) return inv6;
  const int k = 4 + (z > 0 ? 1 : 2 * (int)bc.tlo[xy]) + (z < g.nz - 1 ? 1 : 2 * (int)bc.thi[xy]);
  return T(1) / (T(k) * T(g.ih2));
}

// Same, addressed by the linear cell index e.
template <typename T>
__device__ __forceinline__ T inv_flat(const Geo& g, const Bc<T>& bc, long long e, T inv6) {
  if (g.periodic_z || (e >= g.nxy && e < g.n - g.nxy)) return inv6;
  const int z = e < g.nxy ? 0 : g.nz - 1;
  return inv_diag_unit(g, bc, e - (long long)z * g.nxy, z, inv6);
}

// Solver state in device memory (inside the caller's workspace).
struct Scalars {
  double bb;        // ||b||^2
  double bnorm;     // ||b||
  double rz;        // r.z of the current residual
  double rr;        // ||r||^2
  double alpha;
  double beta;
  double pq;
  double mean_b;    // zero-mean projection of b (singular problems)
  double mean_x;    // mean of the solution (singular problems)
  double rtol;
  double last_rel;  // ||r||/||b|| at the end of the last solve
  long long total_iters;
  int maxit;
  int iter;
  int done;         // 1: the current solve has finished
  int first;        // 1: next p-update is p = z
  int pending;      // 1: x += alpha p still owed
  int zero_x;       // 1: b == 0, the solution is 0
  int status;       // 0 ok, 3 not converged (current solve)
  int pbuf;         // which of the two p buffers holds the latest p
  int nonconv;      // solves that did not converge (per pf_step call)
  int last_iters;
  unsigned ticket;  // last-block counter of the reduction kernels
  int nonfinite;
  unsigned long long sched_next;   // dynamic tile scheduler: next tile
  unsigned sched_done;             // blocks that ran out of tiles
  int zero_solves;                 // solves that ended with no iteration (per pf_step call)
  int max_iters;                   // most iterations of one solve (per pf_step call)
  int solves;                      // solves finished (per pf_step call)
  int short_solves;                // solves that ended after at most one iteration (per pf_step call)
  unsigned bar;                    // arrivals at the barriers of the persistent CG loop
  int timeout;                     // 1: one of its waits ran out (per pf_step call)
  int xzero;                       // 1: the Krylov iterate is the correction of a compensated
                                   // start and is still 0 (its buffer holds stale values)
};

// Operations that are not contracted further: for arithmetic that two kernels
// share bit for bit.
__device__ __forceinline__ float rn_add(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float rn_mul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float rn_fma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double rn_add(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ double rn_mul(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ double rn_fma(double a, double b, double c) { return __fma_rn(a, b, c); }

// ---------------------------------------------------------------- reductions
//
// What a thread sums in FP32 it keeps as an unevaluated pair (hi, lo), and the
// block adds its threads' pairs as pairs; only the block's (or tile's) total
// becomes a double.  The FP64 unit issues one warp instruction in 19 cycles
// per SM (measured: 1.67 thread operations per clock), so converting and
// shuffling doubles in every thread -- 93 FP64 warp instructions per value and
// tile -- cost more than the stencil of a shallow tile: 1.77 kcycles per value
// against about 0.12 for the pairs.  The right-hand side of a 256 x 256 x 64
// film (2048 tiles, three sums) took 78 us that way, the diagnostics (seven
// sums) of 512 x 512 x 64 210 us.

// Sum of a block's threads: a pair of floats (FP32 fields) or a double.
template <typename T>
struct SumOf;
template <>
struct SumOf<double> {
  using type = double;
};
template <>
struct SumOf<float> {
  using type = float2;
};

// (a.x + a.y) + (b.x + b.y) as a normalised pair: TwoSum (Knuth) of the
// leading parts, the rest in the second part; relative error about 2^-46 of
// |a| + |b|.  Past the range of a float the pair is NaN, and the reductions sum
// once more in doubles, as they would the threads' FP32 sums otherwise.
__device__ __forceinline__ float2 pair_add(float2 a, float2 b) {
  const float s = __fadd_rn(a.x, b.x);
  const float z = __fsub_rn(s, a.x);
  float e = __fadd_rn(__fsub_rn(a.x, __fsub_rn(s, z)), __fsub_rn(b.x, z));
  e = __fadd_rn(e, __fadd_rn(a.y, b.y));
  const float h = __fadd_rn(s, e);
  return make_float2(h, __fsub_rn(e, __fsub_rn(h, s)));
}

// Dot-product accumulators.  FP64 fields: plain FMA accumulation.  FP32
// fields: a short run of products (the cells of one vector, closed by run())
// is summed by plain FMAs; the run totals are summed with TwoSum (Knuth), the
// error terms collected in a second float ("cascaded" summation: the
// compensated sum of Ogita, Rump & Oishi, SIAM J. Sci. Comput. 26, 2005,
// applied to runs instead of single products); flush() normalises the pair in
// long loops.  A run of k products carries a relative error of about k u (u =
// 2^-24) of its absolute sum, so with k = 4 the dot keeps close to FP32
// working accuracy of the absolute sum instead of the growth with the length
// of a plain FP32 sum.
template <typename T>
struct Acc;

template <>
struct Acc<double> {
  double s = 0.0;
  __device__ __forceinline__ void add(double a, double b) { s = fma(a, b, s); }
  __device__ __forceinline__ void run() {}
  __device__ __forceinline__ void flush() {}
  __device__ __forceinline__ double sum() const { return s; }
};

template <>
struct Acc<float> {
  float part = 0.f;               // the current run
  float hi = 0.f, lo = 0.f;       // compensated sum of the closed runs
  __device__ __forceinline__ void add(float a, float b) { part = fmaf(a, b, part); }
  __device__ __forceinline__ void run() {
    const float s = __fadd_rn(hi, part);
    const float z = __fsub_rn(s, hi);
    const float se = __fadd_rn(__fsub_rn(hi, __fsub_rn(s, z)), __fsub_rn(part, z));  // hi + part = s + se
    hi = s;
    lo = __fadd_rn(lo, se);
    part = 0.f;
  }
  __device__ __forceinline__ void flush() {
    run();
    const float s = __fadd_rn(hi, lo);
    lo = __fsub_rn(lo, __fsub_rn(s, hi));
    hi = s;
  }
  __device__ __forceinline__ float2 sum() {
    run();
    return make_float2(hi, lo);
  }
};

__device__ __forceinline__ double sum_add(double a, double b) { return a + b; }
__device__ __forceinline__ float2 sum_add(float2 a, float2 b) { return pair_add(a, b); }
__device__ __forceinline__ double sum_xor(double v, int o) { return __shfl_xor_sync(0xffffffffu, v, o); }
__device__ __forceinline__ float2 sum_xor(float2 v, int o) {
  return make_float2(__shfl_xor_sync(0xffffffffu, v.x, o), __shfl_xor_sync(0xffffffffu, v.y, o));
}
__device__ __forceinline__ double warp_total(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ double sum_double(double v) { return v; }
__device__ __forceinline__ double sum_double(float2 v) { return (double)v.x + (double)v.y; }

// Sums of NV values over the NT threads of a block; the sum of value k
// is returned (as a double) in lane 0 of warp k.  Every thread must call it
// with its linear index; it ends without a barrier.  Warp k adds value k of all threads from shared
// memory: 12 additions a value with 256 threads, where a shuffle tree in each
// of the eight warps takes 45.  sm: NV NT elements, 8-byte aligned, that nobody
// else uses until the block's next barrier -- the plane marches lend their
// staging buffers, which are idle between tiles (12 KB of static shared
// memory beside them shrank the L1 and cost k_rhs_w 7 %).  Not inlined: it
// runs once per tile, and its temporaries would count in the march.
template <int NV, int NT, typename V>
__device__ __noinline__ double shared_sums(const V* sm, int tid) {
  const int lane = tid & 31, wid = tid >> 5;
  V d = sm[wid * NT + lane];
#pragma unroll
  for (int j = 1; j < NT / 32; ++j) d = sum_add(d, sm[wid * NT + lane + 32 * j]);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) d = sum_add(d, sum_xor(d, o));
  if constexpr (std::is_same<V, float2>::value) {
    // past the range of a float (or not finite at all): the threads' pairs as doubles
    if (__any_sync(0xffffffffu, !isfinite(d.x))) {
      double e = 0.0;
#pragma unroll 1
      for (int j = 0; j < NT / 32; ++j) e += sum_double(sm[wid * NT + lane + 32 * j]);
      return warp_total(e);
    }
  }
  return sum_double(d);
}
template <int NV, int NT, typename V>
__device__ __forceinline__ double block_sums(const V (&v)[NV], void* scratch, int tid) {
  static_assert(NT % 32 == 0 && NV * 32 <= NT, "a value per warp");
  V* sm = static_cast<V*>(scratch);
  __syncthreads();                 // the scratch may still be read
#pragma unroll
  for (int k = 0; k < NV; ++k) sm[k * NT + tid] = v[k];
  __syncthreads();
  return (tid >> 5) < NV ? shared_sums<NV, NT>(sm, tid) : 0.0;
}

// Block-reduce NV values of one work tile and store them at part[t*NV + k].
// Kernels that hand out tiles dynamically reduce per tile, so the final sum
// (over tiles, in tile order) does not depend on which block ran which tile.
// Must be called by every thread of the block (scratch: see block_sums).
template <int NV, int NT, typename V>
__device__ __forceinline__ void tile_partials(const V (&v)[NV], double* part, long long t, void* scratch) {
  const int tid = threadIdx.x + threadIdx.y * blockDim.x;
  const double d = block_sums<NV, NT>(v, scratch, tid);
  if ((tid & 31) == 0 && (tid >> 5) < NV) part[t * NV + (tid >> 5)] = d;
}

// After every block stored its tile partials: is this the last block to finish?
template <int NT>
__device__ __forceinline__ bool last_block(unsigned* ticket) {
  __shared__ bool last;
  __syncthreads();
  if (threadIdx.x == 0 && threadIdx.y == 0 && threadIdx.z == 0) {
    __threadfence();
    const unsigned t = atomicAdd(ticket, 1u);
    last = (t == gridDim.x - 1);
  }
  __syncthreads();
  return last;
}

// Block-reduce NV values, publish the block's partials, and tell whether this
// block is the last one of the grid to finish (the classic threadfence
// reduction: no block ever waits for another).  Must be called by every
// thread of the block.
template <int NV, int NT = NTHREADS, typename V>
__device__ __forceinline__ bool publish_partials(const V (&v)[NV], double* part, unsigned* ticket) {
  __shared__ V sm[NV * NT];
  tile_partials<NV, NT>(v, part, blockIdx.x, sm);
  return last_block<NT>(ticket);
}

// In the last block: sum the published partials in a fixed order (so results
// are reproducible run to run).
template <int NV, int NT = NTHREADS>
__device__ __forceinline__ void gather_partials(const double* part, long long nblocks, double (&out)[NV],
                                                void* scratch) {
  __shared__ double res[NV];
  const int tid = threadIdx.x + threadIdx.y * blockDim.x;
  double acc[NV];
#pragma unroll
  for (int k = 0; k < NV; ++k) acc[k] = 0.0;
#pragma unroll 1
  for (long long i = tid; i < nblocks; i += NT) {
#pragma unroll
    for (int k = 0; k < NV; ++k) acc[k] += __ldcg(part + i * NV + k);
  }
  const double d = block_sums<NV, NT>(acc, scratch, tid);
  if ((tid & 31) == 0 && (tid >> 5) < NV) res[tid >> 5] = d;
  __syncthreads();
#pragma unroll
  for (int k = 0; k < NV; ++k) out[k] = res[k];
}
template <int NV, int NT = NTHREADS>
__device__ __forceinline__ void gather_partials(const double* part, long long nblocks, double (&out)[NV]) {
  __shared__ double sm[NV * NT];
  gather_partials<NV, NT>(part, nblocks, out, sm);
}

// ------------------------------------------------------------- tile decoding

struct TileCoord {
  int x, y, z0, z1;
  bool active;
};

__device__ __forceinline__ TileCoord tile_coord(const Geo& g, long long t) {
  TileCoord c;
  int ix = (int)(t % g.tiles_x);
  long long r = t / g.tiles_x;
  int iy = (int)(r % g.tiles_y);
  int iz = (int)(r / g.tiles_y);
  c.x = ix * TX + threadIdx.x;
  c.y = iy * TY + threadIdx.y;
  c.z0 = iz * g.tz;
  c.z1 = min(c.z0 + g.tz, g.nz);
  c.active = (c.x < g.nx) && (c.y < g.ny);
  return c;
}

}  // namespace pf
