// Host-only stand-ins for the kernel launchers, linked with the compiled C ABI
// (pf_api) and fake_runtime.cpp: launches are counted and can fail.
// Arguments: a scenario, the solver and what fails
//   fake_cuda solve|noalloc|step|nograph|batch pcg|mg loop|sub|none
// Prints the status, the launches outside and inside captures, and pf_step_info.
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <string>
#include <vector>

#include "pf_internal.h"

extern bool fake_capturing;              // fake_runtime.cpp
extern cudaError_t fake_last;
static std::string failing;
static std::map<std::string, int> direct, captured;

void fake_graph_launch() { direct["graph"] += 1; }
static bool launch(const char* name, bool fails = false) {
  (fake_capturing ? captured : direct)[name] += 1;
  if (fails) fake_last = cudaErrorCooperativeLaunchTooLarge;
  return !fails;
}

// ---------------------------------------------------------------- launchers
namespace pf {
void launch_batch_ramp(const BatchFilm*, int, long long, const BatchState*, cudaStream_t) { launch("ramp"); }
void launch_batch_record(const BatchFilm*, int, int, BatchState*, double*, double*, cudaStream_t) { launch("record"); }
void launch_loop_next(long long*, cudaGraphConditionalHandle, cudaStream_t) { launch("next"); }
void launch_loop_set(long long*, long long, cudaStream_t) { launch("set"); }
int march_blocks_per_sm(int, int) { return 2; }
template <typename T> void launch_rhs_mean(const LaunchCfg&, const Geo&, const Dev<T>&, const T*) { launch("rhs_mean"); }
template <typename T> void launch_rhs(const LaunchCfg&, const Geo&, const Dev<T>& d, const T*, cudaGraphConditionalHandle, int) {
  launch("rhs");
  if (!fake_capturing) d.S->done = d.S->iter = 0;
}
template <typename T> bool launch_cg_loop(const LaunchCfg&, const Geo&, const Dev<T>& d, bool dry) {
  if (dry) return true;
  if (!launch("cg_loop", failing == "loop")) return false;
  if (!fake_capturing) d.S->done = d.S->iter = 1;
  return true;
}
template <typename T> int cg_loop_blocks(const LaunchCfg&, const Geo&, int* small) { return *small = 1, 10; }
template <typename T> void launch_cg_halves(const LaunchCfg&, const Geo&, const Dev<T>&, cudaGraphConditionalHandle) { launch("cg_halves"); }
template <typename T> void launch_cg_p(const LaunchCfg&, const Geo&, const Dev<T>&, int, int, int) { launch("cg_p"); }
template <typename T> void launch_cg_r(const LaunchCfg&, const Geo&, const Dev<T>& d, int, cudaGraphConditionalHandle, int) {
  launch("cg_r");
  if (!fake_capturing) d.S->done = d.S->iter = 1;
}
template <typename T> void launch_cg_finish(const LaunchCfg&, const Geo&, const Dev<T>& d, int) { launch("cg_finish"); }
template <typename T> void launch_sub_mean(const LaunchCfg&, const Geo&, const Dev<T>&) { launch("sub_mean"); }
template <typename T> void launch_invdiag(const LaunchCfg&, const Geo&, const Dev<T>&) { launch("invdiag"); }
template <typename T> void launch_extrap(const LaunchCfg&, long long, T*, T* const[3], long long*, unsigned*, int) { launch("extrap"); }
template <typename T> void launch_tdgl(const LaunchCfg&, const Geo&, const Dev<T>&, const T*, T*, const double*, int, const Noise&) { launch("tdgl"); }
template <typename T> void launch_tdgl_adj(const LaunchCfg&, const Geo&, const Dev<T>&, const T*, T*, const T*, const T*, const double*, double*,
                                           double*, double*) { launch("tdgl_adj"); }
template <typename T> void launch_diag(const LaunchCfg&, const Geo&, const Dev<T>&, const T*, const double*, double*) { launch("diag"); }
template <typename T> void launch_true_residual(const LaunchCfg&, const Geo&, const Dev<T>&, const T*, int, double*) { launch("true_res"); }
template <typename T> bool mg_fused_post(const MgView<T>&) { return false; }
template <typename T> int launch_mg_pre(const LaunchCfg&, const MgView<T>&, Scalars*) { return launch("mg_pre"), 1; }
template <typename T> int launch_mg_rr(const LaunchCfg&, const MgView<T>&, const MgView<T>&, Scalars*) { return launch("mg_rr"), 1; }
template <typename T> int launch_mg_prr(const LaunchCfg&, const MgView<T>&, const MgView<T>&, Scalars*, const std::function<void(int)>&) { return 0; }
template <typename T> int launch_mg_pp(const LaunchCfg&, const MgView<T>&, const MgView<T>&, T*, T*, double*, Scalars*,
                                       const std::function<void(int)>&) { return launch("mg_pp"), 1; }
template <typename T> cudaError_t launch_mg_sub(const LaunchCfg&, const MgTail&, int, const void*, const double*, int, double*, Scalars*) {
  return launch("mg_sub", failing == "sub") ? cudaSuccess : fake_last;
}
template <typename T> int launch_coarse_inverse(const LaunchCfg&, const MgView<T>&, int, double*) { return launch("inverse"), 1; }
template <typename T> int launch_mg_post1(const LaunchCfg&, const MgView<T>&, const MgView<T>&, Scalars*) { return launch("mg_post1"), 1; }
template <typename T> int launch_mg_post2(const LaunchCfg&, const MgView<T>&, int, double*, Scalars*) { return launch("mg_post2"), 1; }
template <typename T> void launch_mg_eps_level(const LaunchCfg&, const MgView<T>&, const MgView<T>&, T*, T*) { launch("mg_eps"); }

#define FAKE(T)                                                                                                   \
  template void launch_rhs_mean<T>(const LaunchCfg&, const Geo&, const Dev<T>&, const T*);                        \
  template void launch_rhs<T>(const LaunchCfg&, const Geo&, const Dev<T>&, const T*, cudaGraphConditionalHandle, int); \
  template bool launch_cg_loop<T>(const LaunchCfg&, const Geo&, const Dev<T>&, bool);                             \
  template int cg_loop_blocks<T>(const LaunchCfg&, const Geo&, int*);                                             \
  template void launch_cg_halves<T>(const LaunchCfg&, const Geo&, const Dev<T>&, cudaGraphConditionalHandle);     \
  template void launch_cg_p<T>(const LaunchCfg&, const Geo&, const Dev<T>&, int, int, int);                       \
  template void launch_cg_r<T>(const LaunchCfg&, const Geo&, const Dev<T>&, int, cudaGraphConditionalHandle, int); \
  template void launch_cg_finish<T>(const LaunchCfg&, const Geo&, const Dev<T>&, int);                            \
  template void launch_sub_mean<T>(const LaunchCfg&, const Geo&, const Dev<T>&);                                  \
  template void launch_invdiag<T>(const LaunchCfg&, const Geo&, const Dev<T>&);                                   \
  template void launch_extrap<T>(const LaunchCfg&, long long, T*, T* const[3], long long*, unsigned*, int);       \
  template void launch_tdgl<T>(const LaunchCfg&, const Geo&, const Dev<T>&, const T*, T*, const double*, int, const Noise&); \
  template void launch_tdgl_adj<T>(const LaunchCfg&, const Geo&, const Dev<T>&, const T*, T*, const T*, const T*, const double*, \
                                   double*, double*, double*);                                                    \
  template void launch_diag<T>(const LaunchCfg&, const Geo&, const Dev<T>&, const T*, const double*, double*);    \
  template void launch_true_residual<T>(const LaunchCfg&, const Geo&, const Dev<T>&, const T*, int, double*);     \
  template bool mg_fused_post<T>(const MgView<T>&);                                                               \
  template int launch_mg_pre<T>(const LaunchCfg&, const MgView<T>&, Scalars*);                                    \
  template int launch_mg_rr<T>(const LaunchCfg&, const MgView<T>&, const MgView<T>&, Scalars*);                   \
  template int launch_mg_prr<T>(const LaunchCfg&, const MgView<T>&, const MgView<T>&, Scalars*, const std::function<void(int)>&); \
  template int launch_mg_pp<T>(const LaunchCfg&, const MgView<T>&, const MgView<T>&, T*, T*, double*, Scalars*,   \
                               const std::function<void(int)>&);                                                  \
  template cudaError_t launch_mg_sub<T>(const LaunchCfg&, const MgTail&, int, const void*, const double*, int, double*, Scalars*); \
  template int launch_coarse_inverse<T>(const LaunchCfg&, const MgView<T>&, int, double*);                        \
  template int launch_mg_post1<T>(const LaunchCfg&, const MgView<T>&, const MgView<T>&, Scalars*);                \
  template int launch_mg_post2<T>(const LaunchCfg&, const MgView<T>&, int, double*, Scalars*);                    \
  template void launch_mg_eps_level<T>(const LaunchCfg&, const MgView<T>&, const MgView<T>&, T*, T*);
FAKE(float)
FAKE(double)
}  // namespace pf

// ----------------------------------------------------------------- scenario
static void print(const char* name, const std::map<std::string, int>& m) {
  std::printf("%s", name);
  for (auto& kv : m) std::printf(" %s=%d", kv.first.c_str(), kv.second);
  std::printf("\n");
}

int main(int argc, char** argv) {
  if (argc != 4) return 2;
  const std::string what = argv[1];
  pf_params p{};
  p.nx = p.ny = 16;
  p.nz = 8;
  p.dx = 1.0;
  p.dt = 0.01;
  p.poisson_rtol = 1e-8;
  p.poisson_maxit = 50;
  p.solver = std::strcmp(argv[2], "mg") ? PF_PCG_JACOBI : PF_PCG_MG;
  p.flags = what == "nograph" ? PF_FLAG_NO_GRAPHS : 0;
  const size_t n = 16 * 16 * 8, bytes = pf_workspace_bytes(&p);
  const int nf = what == "batch" ? 2 : 1;
  std::vector<pf_ctx*> films;
  for (int i = 0; i < nf; ++i) {
    pf_ctx* c = nullptr;
    if (pf_create(&p, nullptr, &c) != PF_OK) return 3;
    if (pf_bind(c, std::calloc(3 * n, 8), std::calloc(n, 8), nullptr, std::aligned_alloc(256, (bytes + 255) / 256 * 256), bytes) != PF_OK)
      return 4;
    films.push_back(c);
  }
  failing = argv[3];
  pf_step_info info{};
  for (int call = 0; call < 2; ++call) {             // the second call knows what the first one met
    direct.clear();
    captured.clear();
    pf_status st;
    if (what == "solve") {
      st = pf_solve_potential(films[0], &info);
    } else if (what == "noalloc") {
      st = pf_solve_potential_noalloc(&p, nullptr, std::calloc(3 * n, 8), std::calloc(n, 8), nullptr, nullptr, nullptr, nullptr, &info);
    } else if (what == "batch") {
      static pf_batch* b = nullptr;
      const size_t bb = pf_batch_workspace_bytes(nf, 4);
      if (!b && pf_batch_create(films.data(), nf, std::aligned_alloc(256, (bb + 255) / 256 * 256), bb, 4, 1, &b) != PF_OK) return 5;
      st = pf_batch_step(b, 1 + 4 * call, &info);
    } else {
      st = pf_step(films[0], 1 + 4 * call, &info);
    }
    std::printf("status %d graph_steps %lld\n", (int)st, (long long)info.graph_steps);
    print("direct", direct);
    print("captured", captured);
  }
  return 0;
}
