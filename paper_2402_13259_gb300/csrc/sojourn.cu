// sojourn.cu -- euler_net_sojourn: sojourn times of tagged customers (Sec. 6,
// Algorithm 4, with the conditional stay probability of Lemma 3), sampled
// while the Euler time loop runs.  The persistent form's slot kernel
// (tile_slots.cuh) advances the customers, or the HBM form's per-step kernels
// (hbm_step.cuh), with the same results.
//
// Algorithm 4 reads, for each step after the customer's entry, the values
// that step produced at the customer's station: the departure draw's input x
// and output D, the post-update count N and the routed counts R_e.  Instead
// of storing whole sample paths and replaying them, the kernels keep the
// tagged customers' state and advance a customer where its station draws the
// step the customer is due in.  The outputs are those of Algorithm 4 run over
// the stored paths, step for step.
//
// A tagged customer has a station and the step it is due in, a place (> 0
// while waiting, 0 in service) and the steps accounted so far:
//   setup at station i after step tau: pos = max(N_tau,i, 1); wait if pos > m_i
//   waiting, step tau:  pos -= D_tau,i; in service from the next step once pos <= m_i
//   service, step tau:  stay with probability Lemma 3 (x_tau,i, D_tau,i, m_i):
//                       u < p_stay, u the first uniform of stream (seed,
//                       purpose 3, slot s, step tau, replication); otherwise
//                       the customer is departure k = floor(w D / 2^32) (w the
//                       stream's second word) of the step's D, which go to the
//                       row's edges in CSR order (R_e each) and then exit.
// m_i is the staffing of the step whose values are read.
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <new>

#include <cuda_runtime.h>

#include "handle.h"
#include "internal.h"

namespace eulernet {
namespace {

int fail(int code, const char* msg) {
  set_last_error(msg);
  return code;
}

int cuda_fail(cudaError_t e, const char* where) {
  cudaGetLastError();  // reported here, not by a later launch check
  char buf[256];
  std::snprintf(buf, sizeof buf, "%s: %s", where, cudaGetErrorString(e));
  set_last_error(buf);
  return e == cudaErrorMemoryAllocation ? EULER_ERR_OOM : EULER_ERR_CUDA;
}

}  // namespace
}  // namespace eulernet

using namespace eulernet;

extern "C" int euler_net_sojourn(euler_net* h, int32_t scheme, double dt, double T, int64_t R,
                                 uint64_t seed, int64_t rep_begin, int32_t station, int64_t tau0,
                                 int32_t samples, int32_t* sojourn, int64_t* stats, void* stream) try {
  if (!h) return fail(EULER_ERR_ARG, "handle is NULL");
  if (scheme != EULER_BACKWARD && scheme != EULER_FORWARD) return fail(EULER_ERR_ARG, "unknown scheme");
  if (!(dt > 0.0) || !(T > 0.0) || !std::isfinite(dt) || !std::isfinite(T))
    return fail(EULER_ERR_ARG, "dt and T must be finite and > 0");
  if (R < 0 || rep_begin < 0) return fail(EULER_ERR_ARG, "replications and rep_begin must be >= 0");
  if (rep_begin + R > (int64_t)1 << 32) return fail(EULER_ERR_TOO_LARGE, "replication index beyond 2^32");
  const int64_t K = euler_num_steps(dt, T);
  if (K >= (1 << 24)) return fail(EULER_ERR_TOO_LARGE, "too many steps (T/dt >= 2^24)");
  if (station < 0 || station >= h->n) return fail(EULER_ERR_ARG, "entry station out of range");
  if (tau0 < 1 || tau0 > K) return fail(EULER_ERR_ARG, "entry step must be in [1, K]");
  if (samples < 1 || samples > (1 << 16)) return fail(EULER_ERR_ARG, "samples must be in [1, 65536]");
  if (R > 0 && !sojourn) return fail(EULER_ERR_ARG, "sojourn output is NULL");
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  cudaError_t e;
  if (!h->d_col && h->E > 0) {
    e = cudaMalloc(&h->d_col, sizeof(int32_t) * (size_t)h->E);
    if (e != cudaSuccess) return cuda_fail(e, "edge table");
    e = cudaMemcpy(h->d_col, h->col.data(), sizeof(int32_t) * (size_t)h->E, cudaMemcpyHostToDevice);
    if (e != cudaSuccess) return cuda_fail(e, "edge table upload");
    h->h2d_bytes += (int64_t)sizeof(int32_t) * h->E;
  }
  const size_t len = (size_t)euler_stats_len(h->n, R);
  if (!stats) {
    if (len > h->sstats_cap) {
      cudaFree(h->d_sstats);
      h->d_sstats = nullptr;
      h->sstats_cap = 0;
      e = cudaMalloc(&h->d_sstats, sizeof(int64_t) * len);
      if (e != cudaSuccess) return cuda_fail(e, "statistics scratch");
      h->sstats_cap = len;
    }
    stats = h->d_sstats;
  }
  int rc = prepare_step_tables(h, dt, T, s);
  if (rc) return rc;
  e = cudaMemsetAsync(stats, 0, sizeof(int64_t) * len, s);
  if (e != cudaSuccess) return cuda_fail(e, "statistics clear");
  if (R == 0) return EULER_OK;
  RunParams p;
  std::memset(&p, 0, sizeof p);
  p.p0 = h->d_p0;
  p.lam = h->d_lam;
  p.h = (float)dt;
  p.K = (int32_t)K;
  p.key0 = (uint32_t)seed;
  p.key1 = (uint32_t)(seed >> 32);
  set_round_keys(p.rk, p.key0, p.key1);
  p.R = R;
  p.rep_begin = rep_begin;
  p.scheme = scheme;
  p.cap = h->opt[EULER_OPT_SAMPLER_CAP] > 0 ? (int32_t)h->opt[EULER_OPT_SAMPLER_CAP] : 1000;
  p.stats = stats;
  p.err = h->d_err;
  p.wait_limit = (int64_t)1 << 25;
  p.muh = h->d_muh;
  p.dep_mode = h->dep_mode();
  p.mtab = h->mtab();
  // The form as for euler_net_simulate; in the HBM form the customers' state
  // lives in global memory and the warp of a customer's station advances it.
  const int forced = (int)h->opt[EULER_OPT_FORM];
  SlotPlan sp;
  const bool tiled = plan_slots(h, scheme, R, false, samples, 0, 0, &sp);
  const bool large = (int64_t)h->n * R >= kHbmMinUnitsPerStep;
  // the documented limit of a small run (and of form 1): one replication's state
  // with its station sums, one step's inputs and departures, and its customers
  const int64_t least = 288 + 60 * (int64_t)h->n + 4 * (int64_t)h->E + 12 * (int64_t)samples;
  if (forced != 2 && (forced > 0 || !large) && least > h->smem_optin)
    return fail(EULER_ERR_TOO_LARGE, "sojourn tile does not fit in shared memory");
  if (forced == 2 || !tiled || (forced <= 0 && takes_hbm(h, R, sp, s))) {
    const int64_t ld = hbm_ld(R);
    const size_t need = (size_t)samples * (size_t)ld;
    if (need > h->cust_cap) {
      cudaFree(h->d_cloc);
      cudaFree(h->d_cpos);
      cudaFree(h->d_csteps);
      h->d_cloc = nullptr;
      h->d_cpos = h->d_csteps = nullptr;
      h->cust_cap = 0;
      e = cudaMalloc(&h->d_cloc, sizeof(unsigned long long) * need);
      if (e == cudaSuccess) e = cudaMalloc(&h->d_cpos, sizeof(int32_t) * need);
      if (e == cudaSuccess) e = cudaMalloc(&h->d_csteps, sizeof(int32_t) * need);
      if (e != cudaSuccess) return cuda_fail(e, "sojourn customer state");
      h->cust_cap = need;
    }
    // EULER_OPT_BLOCK as for euler_net_grad
    const bool own_block = forced == 2 || (forced <= 0 && large);
    const int block = own_block && h->opt[EULER_OPT_BLOCK] > 0 ? (int)h->opt[EULER_OPT_BLOCK] : kHbmBlock;
    if (block % 32 || block > 256) return fail(EULER_ERR_ARG, "HBM-form block must be a multiple of 32 <= 256");
    p.tile_reps = 32;
    p.num_tiles = (R + 31) / 32;
    HbmExtra x;
    x.mode = kHbmSojourn;
    x.cloc = h->d_cloc;
    x.cpos = h->d_cpos;
    x.csteps = h->d_csteps;
    x.col = h->d_col;
    x.S = samples;
    x.station = station;
    x.tau0 = (int32_t)tau0;
    x.out = sojourn;
    return run_hbm_form(h, h->tables(), p, block, s, x);
  }
  p.soj.col = h->d_col;
  p.soj.out = sojourn;
  p.soj.station = station;
  p.soj.tau0 = (int32_t)tau0;
  p.soj.S = samples;
  return run_slots(h, p, kSlotSojourn, sp, (int)std::min<int64_t>(h->sm_count, sp.tiles), s);
} catch (const std::bad_alloc&) {
  return fail(EULER_ERR_OOM, "host memory allocation failed");
} catch (...) {
  return fail(EULER_ERR_CUDA, "unexpected error");
}
