// tile_slots.cuh -- one tile of replications of the persistent shared-memory
// form, run slot by slot: the whole time loop of Algorithm 2 (backward) or
// Algorithm 3 (forward) for Rt replications of one network with the state in
// shared memory.  Shared by the persistent and the batched kernel.
//
// Slots.  Backward, slot tau = 1 .. K+1: every station gathers its routed
// counts of step tau-1 (ring slot (tau-1) % 2) and completes N_{tau-1}, then
// draws step tau from it into ring slot tau % 2.  Forward, slot tau = 1 ..
// K+L-1: the station at level l runs step tau - l, so its predecessors ran
// that step and it ran its own previous step in earlier slots; routed counts
// of step s stay in ring slot s % ring until their consumer has read them.
//
// What bounds it is instruction issue, and the lanes that wait: a unit with
// x > m needs an Erlang time and its binomial's constants, several times the
// work of a unit with x <= m, and on the 100-station DAG 13% of the units are
// such, spread so that 70% of warps of 32 replications of one station hold at
// least one.  So each slot has two phases (unless the plan draws all units in
// place, see plan_slots).  Phase 0 takes the units of the
// tile 32 to a warp, draws those with x <= m to the end and lists the others
// in shared memory; phase 1 takes the list 32 to a warp.  One copy of the
// drawing code serves both.
//
// Units are numbered station position x Rt + replication, and a warp takes
// `task_lanes` consecutive ones, so a tile may have any number of
// replications (a tile count that divides evenly over the SMs) and a small
// run can spread its units over more warps, one or a few to each.  Stations
// are ordered by external arrivals, flow and out-degree, so that the units of
// a warp draw from similar distributions (against level order, forward: 137 ->
// 125 ms with 66 replications to a tile, 403 -> 348 ms with 5 of 2,000
// stations).
//
// Statistics: a unit adds its counts to its own 64-bit sums in global memory
// (reductions without a return value, one address per lane, coalesced); the
// tile's end sums them over replications and over stations.  Against warp
// reductions and per-replication sums in each slot this takes no shuffles and
// leaves the lanes of a warp free to belong to several stations.
//
// Measured on GB300 against the form it replaces in each case (same samplers):
// 100-station DAG, 10,000 replications x 10,000 steps, backward 533 -> 347 ms
// (per-step kernels), 1,237 replications, both schemes 141 -> 45 ms and
// three-station tandem, 1,000 replications 17.3 -> 6.0 ms (a CTA per 32
// replications, a station per warp).  It issues 27 warp instructions per unit
// in 78% of the issue slots, 22.7 of 32 lanes busy (per-step kernels: 41, 61%,
// 19).  Records with three in-edges and shared memory by 32-bit offsets:
// backward 329 -> 323 ms, 2,000 stations s = 10 221 -> 212 ms.
// Tried and slower: the two phases of two halves of the replications in one
// interval, one barrier instead of two (backward 323 -> 342 ms: the interval's
// state costs registers that the draws need); a reduction of X where X = 0
// instead of a branch around it (forward 116.0 -> 117.5 ms).
#pragma once

#include <cstdint>

#include "internal.h"
#include "sampling.cuh"
#include "sojourn_step.cuh"
#include "unit.cuh"

namespace eulernet {

// Dynamic shared memory of the slot kernels (see slot_smem_bytes), addressed
// by 32-bit word offsets: 1/k table [64] | counters [16] | racc i64 [Rt][4],
// the replications' sums at the tile's end | N u32 [n][Rt], the state |
// R i32 [ring][E+1][Rt], routed counts (two ring slots backward, t.ring forward),
// row E zero (stands in for an in-edge that is not there) | aex i32 [n_ex][Rt],
// this slot's arrivals of listed units (backward) | list u16 [n Rt] | GRAD: mu_acc f64 [n][Rt], th_acc f64
// [n_ex][Rt][3], score sums | SOJ: tagged customers' words u64, places i32 and
// step counts i32, [S][Rt] each.
extern __shared__ __align__(16) uint32_t slot_smem[];

__device__ __forceinline__ void slot_add(unsigned long long* a, uint32_t v) {
  if (v) atomicAdd(a, (unsigned long long)v);
}

// acc: global scratch of the CTA, [4][n][Rt] sums of N, max(N - m, 0), D, X,
// then [n_ex][Rt] of A.  rk: the Philox round keys in the kernel's parameter
// space (or shared memory).
// SOJ: the tagged customers of Algorithm 4 (see hbm_step.cuh) act where the
// unit of their station has drawn the step they are due in: a setup reads the
// state after the step, a waiting or service step the step's departure input,
// departures and routed counts.  A unit of another station may read a word
// while it is rewritten in the same phase; it then sees another station or a
// step it is not drawing, and a word is read and written whole (64 bits).
// 100-station DAG, 10,000 replications, 4 customers each, 2,000 steps: 118 ms
// in the per-step kernels -> 65 ms; 162 stations, 102 replications, one step
// at a time with a barrier after each level 161 -> 18 ms for 3,220 steps.
//
// RES: each warp draws one and the same task in every slot (all units in place,
// no more tasks than warps), so its units' records and states stay in
// registers and a slot has no queue and no list.  Such runs are bound by the
// latency of one unit's draws, 2 to 3 us a slot (three-station tandem, 1,000
// replications, 2,402 slots 6.3 -> 5.0 ms; 100 stations, 1,237 replications,
// both schemes 43 -> 40 ms).
template <int SCHEME, bool GRAD, bool EXT, bool SOJ, bool RES>
__device__ __forceinline__ void tile_slots(const NetTables& t, const RunParams& p, int64_t tile,
                                           unsigned long long* const acc, SamplerCtx& cx,
                                           const uint32_t* rk) {
  const int32_t n = t.n;
  const int64_t r0 = tile * p.tile_reps;
  const int Rt = (int)(p.R - r0 < p.tile_reps ? p.R - r0 : p.tile_reps);
  const int U = n * Rt;
  const int L = p.task_lanes;
  const uint32_t magic = Rt > 1 ? 0xFFFFFFFFu / (uint32_t)Rt + 1u : 0u;  // q / Rt = umulhi(q, magic), q < 2^16
  const int tid = threadIdx.x, nthr = blockDim.x;
  const int lane = tid & 31, warp = tid >> 5, nwarps = nthr >> 5;
  const uint32_t rep0 = (uint32_t)(p.rep_begin + r0);
  // word offsets of the area
  const int ring = SCHEME == 0 ? 2 : t.ring;
  const int ring_stride = (t.E + 1) * Rt;
  const int oRacc = 80, oN = oRacc + 8 * Rt, oR = oN + U, oAex = oR + ring * ring_stride;
  const int oList = oAex + t.n_ex * Rt, oMu = (oList + (U + 1) / 2 + 3) / 4 * 4;
  int* const ctr = reinterpret_cast<int*>(slot_smem + 64);
  uint16_t* const list = reinterpret_cast<uint16_t*>(slot_smem + oList);
  double* const mu_acc = reinterpret_cast<double*>(slot_smem + oMu);
  double* const th_acc = mu_acc + U;
  const int S = SOJ ? p.soj.S : 0;
  unsigned long long* const cloc = reinterpret_cast<unsigned long long*>(slot_smem + oMu);
  int32_t* const cpos = reinterpret_cast<int32_t*>(cloc + S * Rt);
  int32_t* const csteps = cpos + S * Rt;
  // Setup of customer ci at station i (servers m of step tau) with N = N_{tau,i}.
  auto soj_setup_at = [&](int ci, int32_t i, int32_t tau, int32_t N, int32_t m) {
    const int32_t pos = N < 1 ? 1 : N;
    cpos[ci] = pos > m ? pos : 0;
    cloc[ci] = soj_pack(i, tau + 1, false);
  };

  for (int q = tid; q < U; q += nthr) {
    const int pos = Rt > 1 ? (int)__umulhi((uint32_t)q, magic) : q;
    slot_smem[oN + q] = t.N0 ? (uint32_t)__ldg(t.N0 + __ldg(t.rec + 3 * pos).x) : 0u;
  }
  for (int k = tid; k < ring * Rt; k += nthr) slot_smem[oR + (k / Rt) * ring_stride + t.E * Rt + k % Rt] = 0u;
  for (int k = tid; k < 8 * Rt; k += nthr) slot_smem[oRacc + k] = 0u;
  for (int k = tid; k < 4 * U + t.n_ex * Rt; k += nthr) __stcg(acc + k, 0ull);
  if (SOJ)
    for (int k = tid; k < S * Rt; k += nthr) {
      cloc[k] = soj_pack(p.soj.station, p.soj.tau0, true);
      cpos[k] = csteps[k] = 0;
    }
  if (GRAD) {
    for (int q = tid; q < U; q += nthr) mu_acc[q] = 0.0;
    for (int k = tid; k < 3 * t.n_ex * Rt; k += nthr) th_acc[k] = 0.0;
  }
  // ctr[0..1]: tasks handed out in phase 0 (by slot parity), ctr[2]: in phase
  // 1, ctr[4..6]: listed units (by slot mod 3).  Each is reset in a slot in
  // which no warp can still read its former value.
  if (tid < 8) ctr[tid] = tid < 3 ? nwarps : 0;
  __threadfence();
  __syncthreads();

  const int last = SCHEME == 0 ? p.K + 1 : p.K + t.L - 1;
  int mod_ring = 0, mod3 = 0;
  const int ntask0 = (U + L - 1) / L;
  int4 ra = make_int4(0, 0, -1, 0), rb = make_int4(0, 0, 0, 0), rc = rb;
  int q = 0, r = 0;
  auto load_unit = [&](int unit) {
    q = unit;
    const int pos = Rt > 1 ? (int)__umulhi((uint32_t)q, magic) : q;
    r = q - pos * Rt;
    ra = __ldg(t.rec + 3 * pos);
    rb = __ldg(t.rec + 3 * pos + 1);
    rc = __ldg(t.rec + 3 * pos + 2);
  };
  const bool own = RES && lane < L && warp * L + lane < U;
  uint32_t nres = 0;  // RES: the unit's state
  if (own) {
    load_unit(warp * L + lane);
    nres = slot_smem[oN + q];
  }
  for (int slot = 1; slot <= last; ++slot) {
    mod_ring = mod_ring + 1 == ring ? 0 : mod_ring + 1;
    mod3 = mod3 == 2 ? 0 : mod3 + 1;
    int* const count = ctr + 4 + mod3;
    if (!RES && tid == 0) {
      ctr[(slot + 1) & 1] = nwarps;
      ctr[2] = nwarps;
      ctr[4 + (mod3 == 2 ? 0 : mod3 + 1)] = 0;
    }
    int ntask = ntask0, listed = U;
#pragma unroll 1
    for (int phase = 0; phase < (RES ? 1 : 2); ++phase) {
      int* const next = phase == 0 ? ctr + (slot & 1) : ctr + 2;
#pragma unroll 1
      for (int task = warp; task < ntask;) {
        const int idx = task * L + lane;
        bool act = RES ? own : lane < L && idx < listed;
        bool heavy = false, wait = phase == 1;  // x > m: listed, or drawn here
        int32_t i = 0, tau = 0, ec = -1, m = 0, e0 = 0, e1 = 0;
        int ocur = oR;  // this step's routed counts
        uint32_t y = 0;
        if (act) {
          if (!RES) load_unit(phase == 0 ? idx : list[idx]);
          i = ra.x;
          ec = ra.z;
          m = ra.w;
          e0 = rb.x;
          e1 = rb.y;
          if (SCHEME == 0) {
            tau = slot;
            ocur = oR + (slot & 1) * ring_stride;
          } else {
            tau = slot - ra.y;
            const int rs = mod_ring - rc.y;
            ocur = oR + (rs < 0 ? rs + ring : rs) * ring_stride;
            act = tau >= 1 && tau <= p.K;
          }
          const bool draws = tau <= p.K;
          if (EXT && p.mtab && act && draws) m = __ldg(p.mtab + (int64_t)(tau - 1) * n + i);
          const uint32_t nprev = RES ? nres : slot_smem[oN + q];
          y = nprev;
          if (act && phase == 0) {
            uint32_t A = 0;
            if (ec >= 0 && draws) {
              PhiloxStream arr;
              arr.init(p.key0, p.key1, 0u, (uint32_t)i, (uint32_t)tau, rep0 + (uint32_t)r, rk);
              arr.refill();  // every Poisson draw takes at least one word
              const float lam = __ldg(p.lam + (int64_t)(tau - 1) * t.n_ex + ec);
              A = (uint32_t)poisson(lam, arr, cx);
              slot_add(acc + 4 * (int64_t)U + ec * Rt + r, A);
              if (GRAD && lam > 0.0f) {
                const float garr = (float)(int32_t)A / lam - 1.0f;
                if (!isnan(garr)) {
                  const float* dl = p.dlam + ((int64_t)(tau - 1) * t.n_ex + ec) * 3;
                  double* th = th_acc + (ec * Rt + r) * 3;
                  th[0] += (double)(garr * __ldg(dl + 0));
                  th[1] += (double)(garr * __ldg(dl + 1));
                  th[2] += (double)(garr * __ldg(dl + 2));
                }
              }
            }
            if (SCHEME == 1 ? draws : slot >= 2) {
              // sums held at kTop, beyond which the caller latches an overflow
              constexpr uint32_t kTop = (uint32_t)kStateLimit + 1u;
              const int oin = (SCHEME == 1 ? ocur : oR + ((slot - 1) & 1) * ring_stride) + r;
              uint32_t in = (slot_smem[oin + rb.z * Rt] + slot_smem[oin + rb.w * Rt]) + slot_smem[oin + rc.x * Rt];
              for (int32_t k = 0; k < rc.w; ++k) {
                in = in < kTop ? in : kTop;
                in += slot_smem[oin + __ldg(t.in_edge + rc.z + k) * Rt];
              }
              in = in < kTop ? in : kTop;
              y = SCHEME == 1 ? nprev + A : nprev;
              y = (y < kTop ? y : kTop) + in;
              if (y > (uint32_t)kStateLimit) {
                cx.err |= kErrOverflow;
                y = (uint32_t)kStateLimit;
              }
            }
            if (SCHEME == 0 && slot >= 2) {  // y is N_{slot-1}: its statistics
              const int32_t mp = EXT && p.mtab ? __ldg(p.mtab + (int64_t)(slot - 2) * n + i) : ra.w;
              atomicAdd(acc + q, (unsigned long long)y);
              if (y > (uint32_t)mp) slot_add(acc + U + q, y - (uint32_t)mp);
            }
            heavy = draws && (!EXT || p.dep_mode == 0) && y > (uint32_t)m;
            wait = heavy && (RES || p.task_inline != 0);
            heavy = heavy && !wait;
            act = draws && !heavy;
            if (SOJ && SCHEME == 0 && !draws)  // slot K+1: the last setups
              for (int ci = r; ci < S * Rt; ci += Rt)
                if (cloc[ci] == soj_pack(i, slot - 1, true)) {
                  const int32_t mp = EXT && p.mtab ? __ldg(p.mtab + (int64_t)(slot - 2) * n + i) : ra.w;
                  soj_setup_at(ci, i, slot - 1, (int32_t)y, mp);
                }
            // backward: the state less this step's departures, a listed unit's
            // A kept beside it (its x = y is the state without A)
            if (RES)
              nres = y + (SCHEME == 0 ? A : 0u);
            else if (SCHEME == 0 || heavy)
              slot_smem[oN + q] = y + (SCHEME == 0 ? A : 0u);
            if (SCHEME == 0 && heavy && ec >= 0) slot_smem[oAex + ec * Rt + r] = A;
          } else if (SCHEME == 0 && act && ec >= 0) {
            y -= slot_smem[oAex + ec * Rt + r];
          }
        }
        if (!RES && phase == 0) {
          const unsigned hb = __ballot_sync(kFull, heavy);
          if (hb) {
            int at = 0;
            if (lane == __ffs(hb) - 1) at = atomicAdd(count, __popc(hb));
            at = __shfl_sync(kFull, at, __ffs(hb) - 1);
            if (heavy) list[at + __popc(hb & ((1u << lane) - 1u))] = (uint16_t)q;
          }
        }
        if (act) {
          PhiloxStream svc;
          svc.init(p.key0, p.key1, 1u, (uint32_t)i, (uint32_t)tau, rep0 + (uint32_t)r, rk);
          svc.refill();
          int32_t D = -1, base = 0, nb = (int32_t)y, branch = 0;
          float T = 0.0f, pw = 0.0f;
          BinomConst bc;
          if (wait) {
            const BinomialArgs dep = departure_wait((int32_t)y, m, __ldg(t.mu + i), p.h, svc, cx);
            nb = dep.n;
            bc = dep.c;
            base = dep.base;
            if (GRAD) branch = dep.branch, T = dep.T, pw = dep.p;
          } else {
            bc = as_const(__ldg(p.p0 + i));
            if (EXT && (p.dep_mode == 1 || (p.dep_mode == 2 && (int32_t)y > m))) {
              // Eq. (1) (Eq. (2) for x > m): D = min(x, Poisson(min(x, m) mu h))
              const int32_t b = (int32_t)y < m ? (int32_t)y : m;
              const int32_t S = poisson((float)b * __ldg(p.muh + i), svc, cx);
              D = S < (int32_t)y ? S : (int32_t)y;
            }
          }
          // One binomial call site draws the departure (base >= 0), then the
          // row's edges, each pass with constants loaded at the end of the one
          // before, so the departure's are not live beside them; its sums and
          // the state are written after the loop (in its first pass they cost
          // 8%: 100-station DAG backward 351 against 329 ms).
          int32_t e = e0, rem = 0;
          int orow = ocur + e0 * Rt + r;
          if (EXT && D >= 0) {
            base = -1;
            rem = nb = D;
            if (e < e1) bc = as_const(__ldg(t.qc + e));
          }
#pragma unroll 1
          while (base >= 0 || e < e1) {
            const int32_t v = binomial_c(nb, bc, svc, cx);  // Bin(0, .) draws nothing
            if (base >= 0) {
              rem = base + v;
              base = -1;
              if (GRAD) {
                BinomialArgs dep;
                dep.branch = branch;
                dep.T = T;
                dep.p = pw;
                mu_acc[q] += (double)departure_score(dep, v, (int32_t)y, m, __ldg(t.mu + i), p.h, __ldg(p.p0f + i));
              }
              D = rem;
            } else {
              slot_smem[orow] = (uint32_t)v;
              rem = rem - v;
              ++e;
              orow += Rt;
            }
            nb = rem;
            if (e < e1) bc = as_const(__ldg(t.qc + e));
          }
          if (SCHEME == 0) {
            if (RES)
              nres -= (uint32_t)D;
            else
              slot_smem[oN + q] -= (uint32_t)D;
          } else {
            const uint32_t nn = y - (uint32_t)D;
            if (RES)
              nres = nn;
            else
              slot_smem[oN + q] = nn;
            atomicAdd(acc + q, (unsigned long long)nn);
            if (nn > (uint32_t)m) slot_add(acc + U + q, nn - (uint32_t)m);
          }
          if (SOJ)
            for (int c = 0; c < S; ++c) {
              const int ci = c * Rt + r;
              if ((int32_t)(cloc[ci] >> 32) != i) continue;
              if (SCHEME == 0 && cloc[ci] == soj_pack(i, tau - 1, true)) {
                const int32_t mp = EXT && p.mtab ? __ldg(p.mtab + (int64_t)(tau - 2) * n + i) : m;
                soj_setup_at(ci, i, tau - 1, (int32_t)y, mp);
              } else if (SCHEME == 1 && cloc[ci] == soj_pack(i, tau, true)) {
                soj_setup_at(ci, i, tau, (int32_t)y - D, m);
                continue;
              }
              if (cloc[ci] != soj_pack(i, tau, false)) continue;
              csteps[ci] += 1;
              const int32_t pos = cpos[ci];
              unsigned long long to = soj_pack(i, tau + 1, false);
              if (pos > 0) {  // waiting
                cpos[ci] = pos - D <= m ? 0 : pos - D;
              } else if (D > 0) {
                const float stay = soj_stay((int32_t)y, D, m);
                PhiloxStream cs;
                cs.init(p.key0, p.key1, 3u, (uint32_t)c, (uint32_t)tau, rep0 + (uint32_t)r, rk);
                cs.refill();
                const float u = cs.uniform();
                uint32_t pick = __umulhi(cs.next(), (uint32_t)D);
                if (!(u < stay)) {
                  to = kSojDone;
                  for (int32_t k = e0; k < e1; ++k) {
                    const uint32_t routed = slot_smem[ocur + k * Rt + r];
                    if (pick < routed) {
                      to = soj_pack(__ldg(p.soj.col + k), tau, true);
                      break;
                    }
                    pick -= routed;
                  }
                }
              }
              cloc[ci] = to;
            }
          atomicAdd(acc + 2 * (int64_t)U + q, (unsigned long long)(uint32_t)D);
          slot_add(acc + 3 * (int64_t)U + q, (uint32_t)rem);
        }
        if (RES || ntask <= nwarps) break;
        if (lane == 0) task = atomicAdd(next, 1);
        task = __shfl_sync(kFull, task, 0);
      }
      __syncthreads();
      if (!RES && phase == 0) {
        listed = *count;
        if (listed == 0) break;  // uniform
        ntask = (listed + L - 1) / L;
      }
    }
  }

  if (own) slot_smem[oN + q] = nres;
  // The tile's sums: over replications to the stations, over stations to the
  // replications; N_K from the state.
  __threadfence();
  __syncthreads();
  int64_t* const st_nk = p.stats + 5 * (int64_t)n + 4 * p.R;
  for (int pos = warp; pos < n; pos += nwarps) {
    const int4 ra = __ldg(t.rec + 3 * pos);
    long long s[6] = {0, 0, 0, 0, 0, 0};  // Q, B, D, X, A, N_K
    for (int r = lane; r < Rt; r += 32) {
      const int q = pos * Rt + r;
      const long long Q = (long long)__ldcg(acc + q), W = (long long)__ldcg(acc + U + q);
      const long long D = (long long)__ldcg(acc + 2 * (int64_t)U + q), X = (long long)__ldcg(acc + 3 * (int64_t)U + q);
      const long long A = ra.z >= 0 ? (long long)__ldcg(acc + 4 * (int64_t)U + ra.z * Rt + r) : 0;
      unsigned long long* rr = reinterpret_cast<unsigned long long*>(slot_smem + oRacc + 8 * r);
      atomicAdd(rr + 0, (unsigned long long)Q);
      atomicAdd(rr + 1, (unsigned long long)D);
      atomicAdd(rr + 2, (unsigned long long)X);
      if (A) atomicAdd(rr + 3, (unsigned long long)A);
      s[0] += Q;
      s[1] += Q - W;
      s[2] += D;
      s[3] += X;
      s[4] += A;
      s[5] += (long long)slot_smem[oN + q];
    }
#pragma unroll
    for (int k = 0; k < 6; ++k) {
      const long long v = warp_sum64(s[k]);
      if (lane == 0 && v)
        atomicAdd(reinterpret_cast<unsigned long long*>(k < 5 ? p.stats + 5 * (int64_t)ra.x + k : st_nk + ra.x),
                  (unsigned long long)v);
    }
  }
  __syncthreads();
  int64_t* const st_rep = p.stats + 5 * (int64_t)n + 4 * r0;
  for (int k = tid; k < 4 * Rt; k += nthr) st_rep[k] = reinterpret_cast<const long long*>(slot_smem + oRacc)[k];
  if (SOJ)
    for (int k = tid; k < S * Rt; k += nthr) {
      const int r = k / S, ci = (k - r * S) * Rt + r;
      p.soj.out[(r0 + r) * S + (k - r * S)] = cloc[ci] == kSojDone ? csteps[ci] : -csteps[ci];
    }
  if (GRAD) {
    // S_r: mu_i sums, then (a, b, phase) summed over external stations in order
    const int64_t C = (int64_t)n + 3;
    for (int64_t k = tid; k < C * Rt; k += nthr) {
      const int r = (int)(k % Rt);
      const int c = (int)(k / Rt);
      int64_t to;
      double v;
      if (c < n) {
        v = mu_acc[c * Rt + r];
        to = __ldg(t.rec + 3 * c).x;
      } else {
        v = 0.0;
        for (int32_t ec = 0; ec < t.n_ex; ++ec) v += th_acc[(ec * Rt + r) * 3 + (c - n)];
        to = c;
      }
      p.scores[(r0 + r) * C + to] = v;
    }
  }
  __syncthreads();
}

}  // namespace eulernet
