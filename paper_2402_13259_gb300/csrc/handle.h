// handle.h -- the library's network handle (private; shared by the host
// translation units, not part of the public ABI).
#pragma once

#include <cstdint>
#include <vector>

#include <cuda_runtime.h>

#include "../../include/eulernet.h"
#include "internal.h"

struct euler_net {
  int32_t n = 0, E = 0, L = 0, max_level = 0, n_ex = 0;
  std::vector<int32_t> row_ptr, col, servers, lvl_ptr, lvl_station, ex_col, N0;
  std::vector<int32_t> ex_station;  // station of each column of the arrival-mean table
  uint64_t uid = 0;                 // unique per handle in this process
  uint64_t tables_gen = 0;          // bumped whenever the per-step tables' inputs change
  std::vector<double> prob, mu;
  int32_t arr_kind = EULER_ARR_NONE;
  std::vector<double> w, table;
  double a = 0, b = 0, period = 1, phase = 0, tab_dt = 1;
  int32_t table_len = 0;

  void* d_tables = nullptr;  // the immutable tables and the error word, one allocation
  int device = 0, sm_count = 0, smem_optin = 0;
  int32_t *d_lvl_station = nullptr, *d_row_ptr = nullptr, *d_in_ptr = nullptr,
          *d_in_edge = nullptr, *d_servers = nullptr, *d_N0 = nullptr, *d_ex_col = nullptr;
  float4* d_qc = nullptr;
  float* d_mu = nullptr;
  unsigned* d_err = nullptr;

  // staffing schedule (host copy) and its per-step table
  std::vector<int32_t> sv_table;
  int32_t sv_len = 0;
  double sv_dt = 1.0;
  int32_t* d_mtab = nullptr;
  size_t mtab_cap = 0;
  float* d_muh = nullptr;

  // external arrival means of steps win_lo .. win_hi multiplied by win_factor
  // (a perturbation of the coupled gradient; off when win_hi < win_lo)
  int64_t win_lo = 1, win_hi = 0;
  double win_factor = 1.0;

  // per-(dt, T) tables of the last call
  double c_dt = -1.0, c_T = -1.0;
  int32_t c_K = 0;
  float4* d_p0 = nullptr;
  float* d_lam = nullptr;
  size_t lam_cap = 0;

  // likelihood-ratio gradient tables of the last (dt, T) and scratch
  double g_dt = -1.0, g_T = -1.0;
  float* d_p0f = nullptr;
  float* d_dlam = nullptr;
  size_t dlam_cap = 0;
  int64_t* d_gstats = nullptr;
  size_t gstats_cap = 0;
  double* d_gscores = nullptr;
  size_t gscores_cap = 0;
  double* d_gpartial = nullptr;
  size_t gpartial_cap = 0;
  double* d_gmu = nullptr;  // HBM-form gradients: score sums [n][ld]
  size_t gmu_cap = 0;
  double* d_gth = nullptr;  // and [n_ex][3][ld]
  size_t gth_cap = 0;
  unsigned long long* d_cloc = nullptr;  // HBM-form sojourn times: customer state
  int32_t* d_cpos = nullptr;
  int32_t* d_csteps = nullptr;
  size_t cust_cap = 0;

  // scratch of the average scheme
  int64_t* d_avg_b = nullptr;
  int64_t* d_avg_f = nullptr;
  size_t avg_cap = 0;

  // sojourn-time sampler: edge destinations and a statistics scratch
  int32_t* d_col = nullptr;
  int64_t* d_sstats = nullptr;
  size_t sstats_cap = 0;
  // HBM-form state; Redge holds hbm_depth ring slots (skewed forward scheme)
  int32_t *d_N = nullptr, *d_Redge = nullptr, *d_tau = nullptr, *d_pos_level = nullptr;
  int32_t hbm_depth = 0;
  int64_t* d_racc = nullptr;
  int64_t hbm_cap_ld = 0, hbm_cap_R = 0;
  cudaStream_t cap_stream = nullptr;
  // persistent form: station records (NetTables::rec) and the CTAs' per-unit sums
  int4* d_rec = nullptr;
  unsigned long long* d_tacc = nullptr;
  size_t tacc_cap = 0;
  std::vector<unsigned long long*> tacc_old;  // smaller arrays, kept for captured graphs

  int64_t opt[13] = {-1, -1, -1, -1, -1, -1, -1, -1, -1, -1, -1, -1, -1};
  int64_t h2d_bytes = 0;  // host-to-device bytes copied by this handle so far

  // The per-step tables depend on mu, the staffing schedule and the arrival
  // window: after a change they are rebuilt on the next call.
  void invalidate_step_tables() {
    c_dt = c_T = -1.0;
    ++tables_gen;
  }

  int32_t dep_mode() const { return opt[EULER_OPT_DEPARTURE] > 0 ? (int32_t)opt[EULER_OPT_DEPARTURE] : 0; }
  const int32_t* mtab() const { return sv_len > 0 ? d_mtab : nullptr; }

  // Ring slots of routed counts in a tile of the persistent form: a backward
  // slot reads only the one before it.
  int32_t slot_ring(int32_t scheme) const {
    return scheme == EULER_BACKWARD || hbm_depth < 2 ? 2 : hbm_depth;
  }

  eulernet::NetTables tables() const {
    eulernet::NetTables t;
    t.n = n;
    t.E = E;
    t.L = L;
    t.lvl_station = d_lvl_station;
    t.row_ptr = d_row_ptr;
    t.qc = d_qc;
    t.in_ptr = d_in_ptr;
    t.in_edge = d_in_edge;
    t.servers = d_servers;
    t.mu = d_mu;
    t.N0 = N0.empty() ? nullptr : d_N0;
    t.ex_col = d_ex_col;
    t.n_ex = n_ex;
    t.pos_level = d_pos_level;
    t.rec = d_rec;
    t.ring = slot_ring(EULER_FORWARD);
    return t;
  }
};

namespace eulernet {
// Units per step (n R) from which one step has work for the whole GPU, the
// share of the SMs' replication slots in use below which the HBM form is then
// faster than the persistent one, the replications up to which it is faster on
// the largest networks (see hbm_beats_tiles), and its default threads per block.
constexpr int64_t kHbmMinUnitsPerStep = int64_t(1) << 18;
constexpr double kTileMinFill = 0.9;
constexpr int64_t kFewReps = 6;
constexpr int kHbmBlock = 256;
// Bytes of HBM-form state per replication chunk, so that a chunk stays in L2.
constexpr int64_t kHbmL2Budget = int64_t(64) << 20;

// Leading dimension of the HBM form's state of R replications (16-byte rows).
inline int64_t hbm_ld(int64_t R) { return (R + 3) / 4 * 4; }

// What an HBM-form run computes besides the statistics (see HbmMode).
struct HbmExtra {
  int mode = kHbmPlain;
  double* mu_acc = nullptr;            // gradients: score sums, zeroed by the run
  double* th_acc = nullptr;
  unsigned long long* cloc = nullptr;  // sojourn times: customer state [S][ld]
  int32_t* cpos = nullptr;
  int32_t* csteps = nullptr;
  const int32_t* col = nullptr;
  int32_t S = 0, station = 0, tau0 = 0;
  int32_t* out = nullptr;              // [R][S]
  const int32_t* state_in = nullptr;   // checkpoint N_{p.tau0}, [n][R], or nullptr (N0)
  int32_t* state_out = nullptr;        // N_K out, [n][R], or nullptr
  int graph_steps = 0;                 // slots per CUDA graph replay (0: the handle's option)
};

// One call in the HBM form: state set-up, the graph of per-step kernels
// replayed to the horizon, statistics (and scores / sojourn times) out.
int run_hbm_form(euler_net* h, const NetTables& t, const RunParams& p, int block, cudaStream_t s,
                 const HbmExtra& x);

// Launch shape of the persistent form (tile_slots.cuh) for R replications.
struct SlotPlan {
  int Rt = 0, block = 32, lanes = 32;
  bool in_place = false;  // units with x > m drawn in place
  bool resident = false;  // and no more tasks than warps: the kernel's RES variant
  int64_t smem = 0, tiles = 0;
  double fill = 1.0;      // share of the SMs' replication slots in use
  int64_t waves = 1;      // tiles an SM runs one after another
  int32_t customers = 0;  // tagged customers per replication
};
bool plan_slots(const euler_net* h, int32_t scheme, int64_t R, bool grad, int32_t soj, int force_Rt, int force_block, SlotPlan* sp);
bool hbm_beats_tiles(const euler_net* h, int64_t R, const SlotPlan& sp, bool alone = false);
// Whether a call on stream s that could take either form takes the HBM form:
// where that is faster, unless s is being captured (a launch of its graphs is no
// operation of another graph; the persistent form's kernels are).
bool takes_hbm(const euler_net* h, int64_t R, const SlotPlan& sp, cudaStream_t s);
int run_slots(euler_net* h, RunParams p, int mode, const SlotPlan& sp, int grid, cudaStream_t s);

// Whether a plain run of R replications takes the persistent form, with *sp
// its plan, or the HBM form.
bool plan_alone(const euler_net* h, int32_t scheme, int64_t R, SlotPlan* sp);

// A plain simulation call of a network that fills the GPU by itself (the
// batched form's large networks), in the form of plan_alone: tables made
// current for (dt, T); `acc` the persistent form's per-unit sums (HBM form if
// nullptr); `block` threads per step kernel and `graph_steps` slots per graph
// replay (0: default) of the HBM form; at most k_limit steps when k_limit > 0
// (tuning runs).  `stats` must be zeroed by the caller, on stream s.
int simulate_alone(euler_net* h, int32_t scheme, double dt, double T, int64_t R, uint64_t seed,
                   int64_t rep_begin, int64_t* stats, cudaStream_t s, int block, int graph_steps,
                   int64_t k_limit, unsigned long long* acc);

// Per-step mean of the external arrivals of station i over step tau: the
// exact integral of lambda_i over ((tau-1) dt, tau dt] (Sec. 2.1.1), in double.
double step_mean(const euler_net& h, int32_t i, int64_t tau, double dt);
// Set the message euler_net_last_error() returns on this thread.
void set_last_error(const char* msg);
// Make the handle's per-call tables (p0 constants, Lambda) current for
// (dt, T) on stream s; returns an EULER_* code.
int prepare_step_tables(euler_net* h, double dt, double T, cudaStream_t s);

// The per-step tables of a call with step dt, written into host buffers in
// ranges, so that every entry point computes them the same way:
//   p0[k], muh[k] for stations i0 + k (k < cnt): the constants of the x <= m
//     departure probability 1 - e^{-mu_i dt} (Lemma 1) and mu_i dt in float;
//   servers[k * n + i] for steps tau0 + k (k < cnt): the staffing schedule's
//     value at the step's start (needs a schedule);
//   lam[k] for the flat entries j0 + k (k < cnt) of the [K][n_ex] table of
//     external-arrival means (Sec. 2.1.1), the arrival window's factor applied.
void step_p0(const euler_net& h, double dt, int32_t i0, int32_t cnt, float4* p0, float* muh);
void step_servers(const euler_net& h, double dt, int64_t tau0, int64_t cnt, int32_t* servers);
void step_lam(const euler_net& h, double dt, int64_t j0, int64_t cnt, float* lam);
}  // namespace eulernet
