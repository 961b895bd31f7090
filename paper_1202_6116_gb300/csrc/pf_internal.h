// Internal interface between the C ABI (pf_api.cu) and the kernel launchers.
#pragma once

#include <functional>

#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <cmath>

#include "pf.h"
#include "pf_common.cuh"

namespace pf {

constexpr int MAX_GRID = 4096;   // reduction partials are sized for this many blocks
constexpr int MAX_NV = 8;        // values reduced per block or tile
constexpr int MG_MAX_LEVELS = 24;
constexpr int MG_MAX_COARSE = 1024;   // cells of the coarsest multigrid level (solved by its inverse)
// The V-cycle's small levels run as one cluster launch (pf_coarse.cu): from
// the first level of at most mg_sub_cells on; its levels of at most
// mg_solo_cells in one block of the cluster.  FP32 from 131 072 cells on: no
// faster on films, from 524 288 much slower (16 SMs); solo from 4096 / 1024 / 256
// cells: the air film of 512 x 512 x 37 15.86 / 15.69 / 15.76 ms per 4 steps,
// 336 x 216 x 32 predictor-corrector 6.95 / 6.88 / 6.89, a batch of 30 films 16.68
// / 16.58 / 16.66.
inline long long mg_sub_cells(size_t word) { return word == 4 ? 65536 : 16384; }
inline long long mg_solo_cells(size_t word) { return word == 4 ? 1024 : 256; }
// Dynamic shared memory of that launch at most: descriptors and masks of 24 levels, three fields of a coarsest
// level of 1024 cells (FP64) or of solo levels from 1024 cells down (FP32), 34 KB either way.
constexpr int MG_TAIL_SMEM = 40 * 1024;
// A multigrid sweep over a large level whose z faces are not periodic runs as
// two launches: the interior planes [b, nz - b), compiled without the face
// code (fewer registers, more resident blocks), and the two face slabs of b
// planes (the pre-smoother's face code also covers the planes next to a face,
// hence b = 2).  Split: the pre-smoother, the prolongation sweep and the second
// post-sweep below the finest level (the finest one also reduces r.z).  The
// second launch costs about 10 us, which a level pays back from about 2^25
// cells (measured: a 2^27-cell level gains, a 2^24-cell one loses), or from
// 2^23 with a permittivity field, whose face code costs more registers.
constexpr int MG_SPLIT_B = 2;
constexpr long long MG_SPLIT_CELLS = 1LL << 25;
constexpr long long MG_SPLIT_CELLS_EPS = 1LL << 23;
inline bool mg_split_level(long long n, int nz, int periodic_z, int eps) {
  return !periodic_z && nz >= 2 * MG_SPLIT_B + 2 && n >= (eps ? MG_SPLIT_CELLS_EPS : MG_SPLIT_CELLS);
}

constexpr unsigned LOOP_POLLS = 1u << 22;   // polls before a barrier of the persistent CG loop gives up (seconds)
constexpr int PLAN_OCC = 6;      // tilings are planned for up to this many blocks per SM

struct LaunchCfg {
  int grid;            // simple per-cell kernels (TX x TY blocks over tiles)
  dim3 block;
  MarchCfg march;      // plane-march kernels (MTX x MTY blocks): the tiling asked for
                       // (tiled = 1), or dflt
  MarchCfg dflt;       // the planned tiling of the CG operator: what a context reports and
                       // takes as "every kernel plans its own" (tiled = 0)
  int tiled;           // 1: another tiling was set (pf_set_tiling)
  int nsm, word, nx, ny, nz;
  int loop_share = 1;  // virtual blocks per block of the persistent Jacobi-PCG loop
  unsigned loop_polls = LOOP_POLLS;   // (pf_set_wait_limit)
  int loop_halves = 0; // 1: that loop as two launches an iteration (both: films of a batch, see pf_cgloop.cu)
  mutable MarchCfg plan[3][PLAN_OCC];   // planned tilings (ntiles = 0: not yet), see kernel_tiling
  int flat_grid;       // flat vector kernels (FLAT_THREADS blocks, grid-stride)
  cudaStream_t stream;
};

// Compensated potential of an FP32 time series (see k_cg_finish_comp): hi is the
// bound phi, lo the rest of the start (the part of the last solution hi cannot
// hold plus the extrapolation increment), ring the differences of the last
// solutions.  lo == nullptr: off.
template <typename T>
struct Comp {
  T* hi;
  T* lo;
  T* ring[3];
  long long* nsolve;   // solves in the history
  int kcap;            // 1 + the highest extrapolation order
};

// Device views of one context's buffers, typed by the storage precision.
template <typename T>
struct Dev {
  T* phi;            // the Krylov iterate: the potential, or its correction when cp.lo is set
  const T* eps;      // nullptr when eps = 1
  T* invd;           // 1/diag(A), only when eps is bound
  T* r;
  T* p0;
  T* p1;
  T* q;
  T* z;              // preconditioned residual (multigrid mode)
  Bc<T> bc;
  double* part;
  Scalars* S;
  Comp<T> cp;
  unsigned short* plo;   // remainder of a compensated FP32 polarization state (3N bf16), or nullptr
};

// Jacobi weights of the two smoothing sweeps: the reciprocals of the roots of
// the degree-2 Chebyshev polynomial on [b/4, b], b = 1.9, which bound the
// spectrum of diag(A)^-1 A (in [0, 2] for this M-matrix) from below b/4 up,
// i.e. 1/lambda_k with lambda_k = (b + a)/2 + (b - a)/2 cos((2k - 1) pi / 4),
// a = b/4.  The pair damps the upper three quarters of the spectrum (the part
// the coarse grid cannot represent) by |(1 - w1 l)(1 - w2 l)| <= 0.35 on
// [b/4, 2]; weighted Jacobi with 6/7 twice leaves up to 0.51 there.  The
// pre-smoother applies w1 then w2, the post-smoother w2 then w1.
constexpr double MG_OMEGA1 = 0.5912564121058501;
constexpr double MG_OMEGA2 = 1.462658863889015;

// Constants of a level's sweeps with eps = 1, formed on the host: per thread
// they are a division and a dozen operations, and as many again per phase of
// the small levels, on the FP64 unit of each SM (the adjoint of 128 x 128 x 32:
// 55.3 -> 46.0 ms with these and the small levels' d c - S; FP64 256 x 256 x 64
// 8.13 -> 7.68 ms per 4 steps).  On the
// planes away from the z faces the operator is d c - S, d the diagonal and S
// the weighted sum of the neighbours, and a sweep's constants fold into the
// weights:
//   both pre-sweeps from zero  e   = p.kf f + S(p.kx, p.ky, p.kz)
//   one sweep of weight w      out = kc c + kf f + S(kx, ky, kz)
template <typename T>
struct LevelK {
  struct Pre {
    T kf, kx, ky, kz;
  } pre;
  struct Sweep {
    T kc, kf, kx, ky, kz;
  } s1, s2;                // weights omega1, omega2
  T d;                     // the diagonal
  T tab[9];                // 1/diag by the kinds of the z faces (as Bc::itab)
  T scale;                 // 1 / children of a coarse cell
};

// One multigrid level as the kernels see it.
template <typename T>
struct MgView {
  Geo g;              // nx, ny, nz, nxy, n, periodic_z of this level
  T ax, ay, az;       // 1/hx^2, 1/hy^2, 1/hz^2
  int fx, fy, fz;     // coarsening factor to the next level (1 or 2)
  const int8_t* tlo;  // z-face electrode masks of this level
  const int8_t* thi;
  T* f;               // right-hand side (level 0: the CG residual r)
  T* e;               // correction (level 0: z = M^-1 r)
  T* et;              // second buffer of the Jacobi sweeps
  const T* eps;       // cell permittivity of this level (nullptr: eps = 1)
  const T* invd;      // 1/diag of this level's operator (with eps only)
  LevelK<T> k;
  MarchCfg mc;
  int split;          // 1: its split sweeps run as interior + face-slab launches (mg_split_level)
};

template <typename T>
inline void sweep_constants(MgView<T>& v) {
  LevelK<T>& k = v.k;
  for (int i = 0; i < 9; ++i)
    k.tab[i] = T(1) / (T(2) * v.ax + T(2) * v.ay + T(faces_of(i / 3) + faces_of(i % 3)) * v.az);
  k.d = T(2) * (v.ax + v.ay + v.az);
  k.scale = T(1) / T(v.fx * v.fy * v.fz);
  const T w1 = T(MG_OMEGA1) * k.tab[0], w2 = T(MG_OMEGA2) * k.tab[0], w12 = w1 * w2;
  k.pre = {w1 + w2 - w12 * k.d, w12 * v.ax, w12 * v.ay, w12 * v.az};
  k.s1 = {T(1) - w1 * k.d, w1, w1 * v.ax, w1 * v.ay, w1 * v.az};
  k.s2 = {T(1) - w2 * k.d, w2, w2 * v.ax, w2 * v.ay, w2 * v.az};
}

// The small levels of the V-cycle, handled by one cluster (pf_coarse.cu): nl
// levels, those from solo on by the cluster's first block, the coarsest of
// coarse cells.
struct MgTail {
  int nl, solo, coarse;
  int cells;                  // of the first one
  int blob_bytes;             // descriptors and solo masks, a multiple of 16
  int smem_bytes;             // the blob, then the solo levels' f, e, e_tmp
};

// One of those levels, as the kernel reads it (host-filled, see MgTail).
template <typename T>
struct SubDesc {
  int nx, ny, nz, nxy, n, per;
  int fx, fy, fz;             // coarsening factors to the next level
  int off, moff;              // shared memory: element offset of the fields, byte offset of the masks (solo levels)
  float rnx, rny;             // 1 / nx, 1 / ny
  T ax, ay, az;
  T tab[9], diag[9];          // 1/diag and diag with eps = 1, by the kinds of the z faces (as Bc::itab)
  T scale;                    // 1 / (fx fy fz)
  T *f, *e, *et;
  const int8_t *tlo, *thi;
  const T *eps, *invd;
};

template <typename T>
void launch_rhs_mean(const LaunchCfg& L, const Geo& g, const Dev<T>& d, const T* P);
template <typename T>
void launch_rhs(const LaunchCfg& L, const Geo& g, const Dev<T>& d, const T* P, cudaGraphConditionalHandle cond,
                int use_cond);
// mg = 1: the search direction is built from z (multigrid-preconditioned
// CG) instead of r/diag, and k_cg_r leaves r.z and beta to the V-cycle.
// second = 1: the second iteration of a compensated multigrid solve (x still
// 0, not staged; needs eps = 1).
template <typename T>
void launch_cg_p(const LaunchCfg& L, const Geo& g, const Dev<T>& d, int mg, int first = 0, int second = 0);
template <typename T>
void launch_cg_r(const LaunchCfg& L, const Geo& g, const Dev<T>& d, int mg, cudaGraphConditionalHandle cond,
                 int use_cond);
// The whole Jacobi-PCG loop as one launch (pf_cgloop.cu).  Returns false, with
// nothing launched, when the grid does not qualify or the launch is not
// possible here; dry: only whether it is.
template <typename T>
bool launch_cg_loop(const LaunchCfg& L, const Geo& g, const Dev<T>& d, bool dry);
// One iteration of that loop as two launches, with the same bits (in a graph's
// conditional loop); and the blocks of a film's loop when it runs alone (*held: of
// such blocks, as many as the GPU holds at a time).
template <typename T>
void launch_cg_halves(const LaunchCfg& L, const Geo& g, const Dev<T>& d, cudaGraphConditionalHandle cond);
template <typename T>
int cg_loop_blocks(const LaunchCfg& L, const Geo& g, int* held);
// Does a film have a 16-byte vector for each of 512 threads per SM?
inline bool loop_fills(const LaunchCfg& L, const Geo& g) { return g.n * L.word / 16 >= L.nsm * 512LL; }
template <typename T>
void launch_cg_finish(const LaunchCfg& L, const Geo& g, const Dev<T>& d, int singular);
template <typename T>
void launch_sub_mean(const LaunchCfg& L, const Geo& g, const Dev<T>& d);
// Thermal random force of one TDGL launch: amp = sigma sqrt(dt) (0: off),
// the Philox key, the device step counter, and whether this launch (the
// last update of a step) advances the counter.
struct Noise {
  double amp;
  unsigned long long seed;
  long long* step;
  int advance;
};

// coef = {a1, a11, a12, g, dt*L}.  corr = 1: predictor-corrector corrector
// (P is the predicted state; Pn holds P_n on entry and P_{n+1} on exit).
template <typename T>
void launch_tdgl(const LaunchCfg& L, const Geo& g, const Dev<T>& d, const T* P, T* Pn, const double* coef,
                 int corr, const Noise& nz);
template <typename T>
void launch_invdiag(const LaunchCfg& L, const Geo& g, const Dev<T>& d);
// Extrapolated initial guess of a time step's solve (see k_extrap; FP32 time
// series form theirs in k_cg_finish).
template <typename T>
void launch_extrap(const LaunchCfg& L, long long n, T* phi, T* const ring[3], long long* nsolve, unsigned* ticket,
                   int kcap);
// Adjoint update (pf_adjoint.cu): lam_out from lam, the adjoint potential psi
// and the state P; adds the parameter sensitivities to grad[4] and, when
// gv_lo/gv_hi are non-NULL, the face-voltage sensitivities.
template <typename T>
void launch_tdgl_adj(const LaunchCfg& L, const Geo& g, const Dev<T>& d, const T* lam, T* lam_out, const T* psi,
                     const T* P, const double* coef, double* grad, double* gv_lo, double* gv_hi);

// Diagnostics (pf_diag.cu): out[0..6] = sums of P_x, P_y, P_z, [P_x > thr],
// f(P), the squared face differences of P, and P.E(phi); coef = {a1, a11, a12, thr}.
template <typename T>
void launch_diag(const LaunchCfg& L, const Geo& g, const Dev<T>& d, const T* P, const double* coef, double* out);

// Persistent step loops (pf_kernels.cu): the count of loop bodies left, and
// the body's last kernel (counts down, sets the while condition).
void launch_loop_set(long long* left, long long n, cudaStream_t st);
void launch_loop_next(long long* left, cudaGraphConditionalHandle h, cudaStream_t st);

// True residual (pf_diag.cu): out[0] = ||b(P) - A phi||^2, out[1] = ||b(P)||^2,
// out[2] = the first for the compensated potential when d.cp.lo is set (else
// equal to out[0]), in FP64 (b projected to zero mean when singular).  out:
// device, 3 doubles.
// Blocks the host between its two passes when singular.
template <typename T>
void launch_true_residual(const LaunchCfg& L, const Geo& g, const Dev<T>& d, const T* P, int singular, double* out);

// One film of a batch as the batch kernels see it (device table).
struct BatchFilm {
  const void* P[2];        // the film's two polarization buffers (3N each)
  void* volt;              // voltages of the ramped z face (nullptr: no ramp)
  long long n, nxy;
  double amp, period;      // V(s) = amp tri(s / period), s = batch step
  int fp32;
  int pad;
};

// Device state of a batch (in the batch workspace).
struct BatchState {
  long long step;          // batch steps completed
  long long records;       // loop records written (or dropped beyond max_records)
  long long record_every;
  long long max_records;
  unsigned ticket;
  unsigned pad;
};

constexpr int BATCH_REC_BLOCKS = 16;   // blocks per film of the loop record

void launch_batch_ramp(const BatchFilm* films, int nfilms, long long max_nxy, const BatchState* bs,
                       cudaStream_t st);
void launch_batch_record(const BatchFilm* films, int nfilms, int buf, BatchState* bs, double* part, double* hist,
                         cudaStream_t st);

// Resident plane-march blocks (MTX x MTY threads) per SM for this precision.
int march_blocks_per_sm(int fp32, int eps);

// Relative time of a plane-march launch whose tiles are cols columns of tz
// planes (the last one shorter) on nsm SMs with occ resident blocks each.
// A tile costs its planes plus the pipeline's fill and the two halo planes
// (about 3 planes in FP32; FP64 marches are bound by the FP64 unit, which the
// halo planes do not use: half a plane).  The tiles go to the SMs in order,
// each to the first one free (groups of SMs free at the same time are kept
// together); b blocks sharing an SM take 1 + k (b - 1) times as long as one
// alone, k = 0.6 in FP32 and 0.8 in FP64 (fitted to sweeps of the depth).
inline double march_cost(long long cols, int nz, int tz, int nsm, int occ, int word) {
  const double c = word == 4 ? 3.0 : 0.5, k = word == 4 ? 0.6 : 0.8;
  struct Group {
    double t;
    long long m;
  };
  Group q[160];                                   // three are needed: every chunk but the last is equally deep
  int nq = 1;
  q[0] = Group{0.0, nsm};
  auto insert = [&](double t, long long m) {      // groups in ascending order of t
    int i = nq;
    while (i > 0 && q[i - 1].t > t) --i;
    if (i > 0 && q[i - 1].t == t) {
      q[i - 1].m += m;
      return;
    }
    for (int j = nq; j > i; --j) q[j] = q[j - 1];
    q[i] = Group{t, m};
    ++nq;
  };
  double span = 0.0;
  for (int z = 0; z < nz; z += tz) {
    const double d = std::min(tz, nz - z) + c;
    for (long long left = cols; left > 0;) {
      const double t = q[0].t;
      long long m = q[0].m, rounds = 1;
      if (nq == 1 && left > m) rounds = left / m;   // every SM free at once: whole rounds
      m = std::min(m, left);
      if (m == q[0].m) {
        for (int j = 1; j < nq; ++j) q[j - 1] = q[j];
        --nq;
      } else {
        q[0].m -= m;
      }
      insert(t + rounds * d, m);
      span = std::max(span, t + rounds * d);
      left -= m * rounds;
    }
  }
  const double tiles = span / (std::min(tz, nz) + c);      // whole tiles on the busiest SM
  const double full = std::floor(tiles / occ), rest = tiles - full * occ;
  const double f = full * (1.0 + k * (occ - 1)) + (rest <= 1.0 ? rest : 1.0 + k * (rest - 1));
  return span * f / tiles;
}

// Tiling of a plane march over an nx x ny x nz grid: 16 bytes of cells per
// thread when nx allows it, and the tile depth (at most tzmax planes, even for
// even_tz) of least march_cost.  turns > 0: among those of at most two planes, with
// turns tiles per resident block, or whose tiles fill the resident blocks a whole
// number of times but for 6 %.  One rule for every size: a film of 1024 x 1024
// columns takes the deepest tiles, one of 64 x 64 a couple of planes per tile.
// (The rule before it, the deepest of 32 .. 2 planes with three tiles per
// resident block, gave a 256 x 256 x 64 film tiles of 2 planes: 55 us for the
// right-hand side, 33 for the search direction; planned, 37 and 23.)
inline MarchCfg march_cfg(int nx, int ny, int nz, int nsm, int occ, int tzmax, bool even_tz, int word,
                          int turns = 0) {
  MarchCfg m{};
  const int v = 16 / word;
  m.vx = nx % v == 0 ? v : 1;
  const int bx = MTX * m.vx;
  m.tiles_x = (nx + bx - 1) / bx;
  m.tiles_y = (ny + MTY - 1) / MTY;
  const long long cols = (long long)m.tiles_x * m.tiles_y;
  double best = 0.0;
  m.tz = even_tz ? 2 : 1;
  int last = 0;
  for (int tz = std::min(tzmax, nz); tz >= 1; --tz) {
    if (even_tz && (tz & 1)) continue;
    const int chunks = (nz + tz - 1) / tz;
    const long long tiles = cols * chunks, slots = (long long)nsm * occ;
    if (tz > 2 && tiles < turns * slots && 50 * tiles < 47 * ((tiles + slots - 1) / slots * slots)) continue;
    if (chunks > 128) {          // march_cost is a sum over the chunks: very tall grids take a plain rule
      if (best == 0.0) {
        m.tz = tz;
        while (m.tz > 2 && cols * ((nz + m.tz - 1) / m.tz) < 3LL * nsm * occ) m.tz = m.tz / 4 * 2;
      }
      break;
    }
    // of the depths with this many chunks: the deepest, the even split, multiples of 8
    if (chunks == last && (nz + chunks - 1) / chunks != tz && tz % 8 != 0) continue;
    last = chunks;
    const double cost = march_cost(cols, nz, tz, nsm, occ, word);
    if (best == 0.0 || cost < 0.999 * best) {
      best = cost;
      m.tz = tz;
    }
  }
  m.ntiles = cols * ((nz + m.tz - 1) / m.tz);
  m.grid = (int)std::min<long long>(m.ntiles, std::min(MAX_GRID, nsm * occ));
  return m;
}

// Tiling of one plane-march kernel on the fine grid (its shared-memory limit
// already raised; occ caches its occupancy): the one asked for, on its own
// occupancy, or the planned one.  deep: tiles of up to 64 planes (the kernels
// that sum over their tiles), else 32 (the TDGL update on 1024 x 1024 x 128:
// 1.00 ms with 32 planes, 1.02 with 64).  turns: three for the FP32 update with noise,
// whose blocks keep the issue slots busy: two on an SM take nearly twice as long as one,
// which march_cost does not know, so its tiles balance the load or fill the SMs evenly
// (512 x 512 x 64 256 us, 286 without; 256 x 256 x 16 29 and 33; 96 x 96 x 48 17.5 and 20.6).
template <class K>
inline MarchCfg kernel_tiling(K kernel, size_t bytes, const LaunchCfg& L, int& occ, bool deep, int turns = 0) {
  if (occ == 0) {
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kernel, MTX * MTY, bytes) != cudaSuccess) occ = 1;
    cudaGetLastError();
    occ = std::max(occ, 1);
  }
  if (L.tiled) {
    MarchCfg m = L.march;
    const int bps = m.bps > 0 ? std::min(m.bps, occ) : occ;
    m.grid = (int)std::min<long long>(m.ntiles, std::min<long long>(MAX_GRID, (long long)bps * L.nsm));
    return m;
  }
  const int o = std::min(occ, PLAN_OCC);
  MarchCfg& m = L.plan[turns ? 2 : deep ? 1 : 0][o - 1];
  if (m.ntiles == 0) m = march_cfg(L.nx, L.ny, L.nz, L.nsm, o, deep ? 64 : 32, false, L.word, turns);
  return m;
}

// Grid geometry and launch shapes of the fine level for these parameters
// (shared by the context-based entry points and the allocation-free solve).
inline void setup_launch(const pf_params* p, int nsm, cudaStream_t stream, Geo& g, LaunchCfg& L) {
  g = Geo{};
  g.nx = p->nx;
  g.ny = p->ny;
  g.nz = p->nz;
  g.periodic_z = p->periodic_z;
  g.zair = p->nz - p->n_air;
  g.nxy = (long long)g.nx * g.ny;
  g.n = g.nxy * g.nz;
  g.ih = 1.0 / p->dx;
  g.ih2 = g.ih * g.ih;
  g.tiles_x = (g.nx + TX - 1) / TX;
  g.tiles_y = (g.ny + TY - 1) / TY;
  const long long cols = (long long)g.tiles_x * g.tiles_y;
  g.tz = 1;
  for (int tz : {16, 8, 4, 2}) {
    if (cols * ((g.nz + tz - 1) / tz) >= 4LL * nsm) {
      g.tz = tz;
      break;
    }
  }
  g.tiles_z = (g.nz + g.tz - 1) / g.tz;
  g.ntiles = cols * g.tiles_z;
  L = LaunchCfg{};
  const int fp32 = p->precision == PF_FP32;
  L.nsm = nsm;
  L.word = fp32 ? 4 : 8;
  L.nx = g.nx;
  L.ny = g.ny;
  L.nz = g.nz;
  L.march = march_cfg(g.nx, g.ny, g.nz, nsm, std::min(PLAN_OCC, march_blocks_per_sm(fp32, p->has_eps)), 64, false, L.word);
  L.dflt = L.march;
  const long long nvec = (g.n + 3) / 4;
  L.flat_grid = (int)std::max<long long>(
      1, std::min<long long>((nvec + FLAT_THREADS - 1) / FLAT_THREADS, std::min(MAX_GRID, 4 * nsm)));
  L.block = dim3(TX, TY, 1);
  L.grid = (int)std::min<long long>(g.ntiles, std::min(MAX_GRID, 8 * nsm));
  L.stream = stream;
}

// Record the message returned by pf_last_error(NULL) (fixed buffer, no allocation).
void set_global_error(const char* what, const char* detail = nullptr);


// Multigrid V-cycle pieces (pf_mg.cu).
template <typename T>
int launch_mg_pre(const LaunchCfg& L, const MgView<T>& lv, Scalars* S);
template <typename T>
int launch_mg_rr(const LaunchCfg& L, const MgView<T>& lv, const MgView<T>& cv, Scalars* S);
// Pre-smoother and residual of a split FP32 level as one fused pass over its
// interior planes (plus the face slabs' own kernels); returns the launches, 0
// when the level does not qualify (then nothing was launched).
// mark(i) is called after the i-th of its launches (0 .. 2; the profiler's marks).
template <typename T>
int launch_mg_prr(const LaunchCfg& L, const MgView<T>& lv, const MgView<T>& cv, Scalars* S,
                  const std::function<void(int)>& mark);
// Whether the finest level's post-sweeps run fused (launch_mg_pp); then the
// V-cycle keeps the pre-smoothed correction out of z (in z_tmp) and uses ep
// (the CG's q, dead between the residual update and the next search
// direction) for e'.
template <typename T>
bool mg_fused_post(const MgView<T>& lv);
// Prolongation sweep + second post-sweep of the finest level, fused on its
// interior (lv.e: the pre-smoothed correction, ep: e', z: the result; r.z and
// beta as k_mg_post2); returns the launches, 0 when not eligible.
template <typename T>
int launch_mg_pp(const LaunchCfg& L, const MgView<T>& lv, const MgView<T>& cv, T* ep, T* z, double* part,
                 Scalars* S, const std::function<void(int)>& mark);
// The small levels (see MgTail; blob: their descriptors and masks in device
// memory); cinv: the coarsest level's inverse; last: the first of them is the
// finest level (r.z and beta are formed too).
template <typename T>
cudaError_t launch_mg_sub(const LaunchCfg& L, const MgTail& t, int eps, const void* blob, const double* cinv, int last,
                          double* part, Scalars* S);
// Inverse of the coarsest operator into cinv (n^2 doubles, and 2 n of
// scratch after them); returns the launches.
template <typename T>
int launch_coarse_inverse(const LaunchCfg& L, const MgView<T>& C, int singular, double* cinv);
template <typename T>
int launch_mg_post1(const LaunchCfg& L, const MgView<T>& lv, const MgView<T>& cv, Scalars* S);
template <typename T>
int launch_mg_post2(const LaunchCfg& L, const MgView<T>& lv, int last, double* part, Scalars* S);
// Permittivity of a coarse level (the mean of the fine children, into ceps)
// and 1/diag of its operator (into cinvd).
template <typename T>
void launch_mg_eps_level(const LaunchCfg& L, const MgView<T>& fine, const MgView<T>& coarse, T* ceps, T* cinvd);

}  // namespace pf
