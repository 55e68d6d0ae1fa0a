// Host-side state of a tadmm handle and the per-precision / per-dimension
// implementation entry points (explicitly instantiated in tadmm_f64.cu and
// tadmm_f32.cu).
#pragma once

#include <cuda_runtime.h>

#include <algorithm>
#include <string>
#include <vector>

#include "../../include/tadmm.h"
#include "tadmm_device.cuh"

// Scratch of the implicit-KKT backward pass (grown on demand).
struct BwdBufs {
  void *act = nullptr, *cnt = nullptr, *amask = nullptr, *psi = nullptr, *kks = nullptr, *pos0 = nullptr,
       *force = nullptr, *Xp = nullptr, *Up = nullptr, *Wx = nullptr, *Wu = nullptr, *bstat = nullptr,
       *bs = nullptr, *S = nullptr, *vec = nullptr, *gX = nullptr, *gout = nullptr, *xpol = nullptr,
       *piv = nullptr, *ndep = nullptr, *hmask = nullptr, *Wb = nullptr, *pchg = nullptr, *set_act = nullptr,
       *set_W = nullptr;
  size_t act_cap = 0, cnt_cap = 0, amask_cap = 0, psi_cap = 0, kks_cap = 0, pos0_cap = 0, force_cap = 0,
         Xp_cap = 0, Up_cap = 0, Wx_cap = 0, Wu_cap = 0, bstat_cap = 0, bs_cap = 0, S_cap = 0, vec_cap = 0,
         gX_cap = 0, gout_cap = 0, xpol_cap = 0, piv_cap = 0, ndep_cap = 0, hmask_cap = 0, Wb_cap = 0,
         pchg_cap = 0, set_act_cap = 0, set_W_cap = 0;
};

namespace tadmm {

// Estimated work of the persistent kernel's groups: those of at most kGroupMax agents
// ([0]) and the larger scenarios, alone on a CTA ([1]).
inline double group_work(int T, double pairs) { return T * (600.0 + 30.0 * pairs / 32.0); }
struct GroupLoad {
  double sum[2] = {0.0, 0.0}, top[2] = {0.0, 0.0};
  void add(bool large, double w) {
    sum[large] += w;
    top[large] = w > top[large] ? w : top[large];
  }
};

}  // namespace tadmm

struct tadmm_handle {
  int prec = 64, nx = 0, nu = 0, dp = 0, n_scen = 0;
  int64_t tot_on = 0;       // words of the graph mode's partner masks
  int64_t tot_agents = 0, tot_as = 0, tot_ps = 0, tot_xs = 0, tot_pairs = 0;
  tadmm_options opt{};
  std::vector<int32_t> N, T;
  std::vector<tadmm::ScenMeta> meta_h;
  int device = 0, sm_count = 0;

  // device state
  tadmm::ScenMeta* meta = nullptr;
  int32_t* order = nullptr;
  int32_t* goff = nullptr;      // scenario groups of the persistent kernel
  int32_t* gmem = nullptr;
  int32_t* gorder = nullptr;
  int n_groups = 0;
  int max_group_pairs = 0;
  tadmm::GroupLoad load;        // their estimated work
  int32_t* pairs = nullptr;
  int32_t* deg = nullptr;       // [tot_agents] copies per agent
  int32_t* adj_ptr = nullptr;   // [tot_agents + 1]
  int32_t* adj = nullptr;       // listed-pair adjacency (sparse scenarios)
  std::vector<int32_t> pair_count_h, pair_ij_h;  // caller's pair lists (empty: all pairs)
  int32_t* pair_scen = nullptr;
  int32_t* agent_scen = nullptr;
  void* model = nullptr;
  void* Qd = nullptr;
  void* Rd = nullptr;
  void* Qfd = nullptr;
  void* x_init = nullptr;
  void* x_ref = nullptr;
  void* a = nullptr;
  void* w0 = nullptr;
  void* theta = nullptr;
  void* models = nullptr;        // heterogeneous agents: [tot_agents] per-agent model (A, B, umin, umax)
  double* st_models = nullptr;   // their float64 staging
  std::vector<double> models_h;  // host packing of the caller's per-agent A, B (kept for async copies)
  int hetero = 0;                // 1: per-agent dynamics
  void* phi = nullptr;           // over-relaxation: [tot_ps] pair part of the consensus copies
  void* sx = nullptr;            // over-relaxation: [tot_as][dp] agent part of the consensus copies
  void* hprev = nullptr;         // homotopy hot start: [tot_as][dp] previous coupling terms
  void* hmu = nullptr;           //   [tot_as][nu] bound multipliers of the previous optimum
  void* hdmu = nullptr;          //   [tot_as][nu] their segment direction
  void* X = nullptr;
  void* h = nullptr;
  void* U = nullptr;
  void* Us = nullptr;
  void* cache = nullptr;
  uint16_t* Wm = nullptr;
  uint16_t* Cm = nullptr;
  int32_t* status = nullptr;
  int32_t* iters = nullptr;
  int32_t* cur_lvl = nullptr;
  double* res = nullptr;
  unsigned long long* eqp = nullptr;
  unsigned long long* fact = nullptr;
  double* rho_out = nullptr;     // [n_scen] penalty at the end of the last solve
  int32_t* rho_chg = nullptr;    // [n_scen] residual-balancing changes of the last solve
  int32_t* queue = nullptr;

  // float64 staging in the caller's layouts (imports and exports)
  double* st_model = nullptr;   // A, B, umin, umax
  double* st_agent = nullptr;   // Qd, Rd, Qfd, x_init, x_ref (5 blocks)
  double* st_a = nullptr;       // [tot_ps][dp]
  double* st_w0 = nullptr;      // [tot_as][dp]
  double* ex_buf = nullptr;     // export scratch
  double* st_costs = nullptr;   // tadmm_update_costs: float64 staging of Qd, Rd, Qfd, x_ref before validation
  int32_t* cost_flag = nullptr; //   its device-side validation flag
  double* sqp_buf = nullptr;     // tadmm_sqp: [n_scen] objective | [n_scen] min distance | [n_scen] uint8 keep mask
  size_t ex_bytes = 0;

  // plain mode
  int32_t* flag = nullptr;               // device: agent QP failure code
  unsigned long long* red2 = nullptr;    // device: residual maxima bits
  void* pinned = nullptr;                // host pinned readback buffer

  // batched mode launch shape and captured graph
  int tpc = 0, cps = 0, variant = 0;
  int auto_tpc = 0;         // threads per CTA by default_threads (0: not asked for yet)
  int di = 0;               // the shared model is an exact double integrator
  int ax = 0;               // it is, or every agent's own model is axis-separable (tadmm_axis.cuh)
  cudaStream_t cap_stream = nullptr;
  cudaGraphExec_t gexec = nullptr;
  double g_tol = -1.0;
  int g_iter = -1, g_tpc = -1, g_cps = -1, g_var = -1;
  int solved = 0;
  int bwd_polished = 0;     // the backward active set was refined by tadmm_polish after the last solve
  int64_t launches = 0;   // kernel launches enqueued by the last solve
  BwdBufs bwd;

  // graph mode (conditional WHILE node over the per-iteration phase kernels)
  void *gs_iter = nullptr, *gs_active = nullptr, *gs_fail = nullptr, *gs_rb = nullptr,
       *gs_sb = nullptr, *gs_on = nullptr, *gs_done = nullptr;
  void* gs_blk = nullptr;   // int2 (scenario, first agent) per 32-agent gather block
  int n_gblk = 0;
  int gs_ready = 0;         // all of these are allocated and the gather table is uploaded
  cudaGraphExec_t wexec = nullptr;
  double w_tol = -1.0;
  int w_iter = -1;
};

namespace tadmm {

int set_error(int code, const std::string& msg);
int cuda_check(cudaError_t e, const char* what);

// Threads per CTA of the persistent kernel unless given or tuned; resident: CTAs of 128,
// 64 and 32 threads that an SM holds of this batch (asked for only with a large scenario).
//
// Groups of at most 32 agents: an SM holds eight warps of variant 0 (registers), so as
// many threads as still let every group run at once (receding horizon, 256 scenarios:
// 44 ms with 128 threads, 58 with 32; 4096 scenarios, 2223 groups: 361 ms with 32
// threads, 485 with 64, 734 with 128).  The over-relaxed sweep, all pairs in FP64, takes
// 128 (512 scenarios, 150 iterations: 173 ms, 224 with 64, 316 with 32).
//
// With a larger scenario the CTAs hold its pairs in shared memory too, so an SM holds
// fewer of the small ones, and the scenario itself may take longer than all the rest.
// Then the shape of the shortest estimated span: the longest CTA, or all CTAs over the
// slots, where a CTA of 64 (128) threads takes 0.53 (0.41) of the time of one warp for a
// group and 0.53 (0.36) for a large scenario, as measured.  20 iterations, ms with 32 /
// 64 / 128 threads: 1000 small scenarios with one of 64 and one of 200 agents 677 / 346 /
// 190, with one of 90 agents 233 / 143 / 74; 4000 with one of 64 agents 183 / 139 / 183;
// 1500 of 40 agents 98 / 89 / 121; 300 of 33 to 48 agents 124 / 71 / 64, 700 of them
// 131 / 87 / 106.  The estimate takes the fastest of each but the last, where the two
// spans are within 3 % and it takes 128.
inline int default_threads(const GroupLoad& load, int n_groups, bool relaxed, int sm_count, const int (&resident)[3]) {
  const int sm = sm_count > 0 ? sm_count : 1, ng = n_groups > 0 ? n_groups : 1;
  if (load.sum[1] == 0.0) {
    const int fit = 8 * 32 * sm / ng;
    return (fit >= 128 || relaxed) ? 128 : (fit >= 64 ? 64 : 32);
  }
  constexpr int kThreads[3] = {128, 64, 32};
  constexpr double kCost[3][2] = {{0.41, 0.36}, {0.53, 0.53}, {1.0, 1.0}};
  int best = 128;
  double span = 0.0;
  for (int k = 0; k < 3; ++k) {
    if (resident[k] < 1) continue;
    const double* c = kCost[k];
    const double longest = std::max(c[0] * load.top[0], c[1] * load.top[1]);
    const double s = std::max(longest, (c[0] * load.sum[0] + c[1] * load.sum[1]) / ((double)resident[k] * sm));
    if (span == 0.0 || s < span) {
      span = s;
      best = kThreads[k];
    }
  }
  return best;
}

// Graph mode: whether everything after an iteration's x-update runs as one CTA per
// scenario (k_g_tail) and not as grid-wide kernels.  That saves about 5 us of launches
// an iteration and costs about 3.5 ns per pair-step of the largest scenario, so the
// line lies near 2000 of them (measured, one scenario, us an iteration against the
// grid-wide kernels: 14 agents x 20 steps, 1820 pair-steps, -1; 8 x 80, 2240, +4;
// 20 x 20, 3800, +5; 32 x 20, 9920, +16; 32 x 1280, 635 000, +2195).  Agent-steps count
// too: each takes its sum.  With more scenarios than one per SM the CTAs fill the GPU
// and the two are level (256 of 32 agents x 20 steps: -7), unless one of them is longer
// than an SM's share of all.  k_g_tail holds at most kGroupMax agents, the grid-wide
// kernels at most 65535 steps.
constexpr int kTailWork = 2560;
inline bool tail_per_scenario(const std::vector<ScenMeta>& scen, int sm_count) {
  int64_t top = 0, total = 0;
  int nmax = 0, tmax = 0;
  for (const ScenMeta& m : scen) {
    const int64_t work = ((int64_t)m.P + m.N) * m.T;
    top = work > top ? work : top;
    total += work;
    nmax = m.N > nmax ? m.N : nmax;
    tmax = m.T > tmax ? m.T : tmax;
  }
  if (nmax > kGroupMax) return false;
  return top <= kTailWork || top <= total / (sm_count > 0 ? sm_count : 1) || tmax > 65535;
}

// Device blocks of the graph mode: all of them or, after a failed allocation, none
// (the next solve then tries again).
inline void graph_state_free(tadmm_handle* h) {
  void** const blocks[] = {&h->gs_iter, &h->gs_active, &h->gs_fail, &h->gs_rb,
                           &h->gs_sb,   &h->gs_on,     &h->gs_done, &h->gs_blk};
  for (void** p : blocks) {
    if (*p) cudaFree(*p);
    *p = nullptr;
  }
  h->gs_ready = 0;
}

inline int graph_state_alloc(tadmm_handle* h) {
  graph_state_free(h);
  const size_t n = (size_t)h->n_scen;
  const size_t on = (size_t)(h->tot_on > 0 ? h->tot_on : 1), blk = (size_t)(h->n_gblk > 0 ? h->n_gblk : 1);
  struct { void** p; size_t bytes; } const want[] = {
      {&h->gs_iter, 4 * n}, {&h->gs_active, 4 * n}, {&h->gs_fail, 4 * n}, {&h->gs_rb, 8 * n},
      {&h->gs_sb, 8 * n},   {&h->gs_done, 8},       {&h->gs_on, 4 * on},  {&h->gs_blk, 8 * blk}};
  for (const auto& w : want)
    if (cudaMalloc(w.p, w.bytes) != cudaSuccess) {
      cudaGetLastError();
      *w.p = nullptr;
      graph_state_free(h);
      return set_error(TADMM_ENOMEM, "graph-mode state allocation failed");
    }
  return TADMM_OK;
}

template <typename F, int NX, int NU, int DP>
struct Impl {
  static int import_inputs(tadmm_handle* h, cudaStream_t st);
  static int solve_batched(tadmm_handle* h, double tol, int max_iter, cudaStream_t st);
  static int solve_plain(tadmm_handle* h, double tol, int max_iter, cudaStream_t st);
  static int solve_graph(tadmm_handle* h, double tol, int max_iter, cudaStream_t st);
  static int export_solution(tadmm_handle* h, double* X, double* U, double* theta, int8_t* W,
                             cudaStream_t st);
  static int max_ctas_per_sm(int tpc, int variant, const tadmm_handle* h);
  static int backward(tadmm_handle* h, const double* gX_dev, double theta_eps, double* gout_dev, double* xpol_dev,
                      cudaStream_t st);
  static int relinearize(tadmm_handle* h, const uint8_t* keep, cudaStream_t st);
  static int sqp_measure(tadmm_handle* h, double* J, double* dmin, cudaStream_t st);
  static int import_costs(tadmm_handle* h, int which, cudaStream_t st);
  static int polish(tadmm_handle* h, double theta_eps, int max_rounds, double kkt_tol, uint8_t* act_dev, int8_t* W_dev,
                    int32_t* status, int32_t* rounds, cudaStream_t st);
};

}  // namespace tadmm
