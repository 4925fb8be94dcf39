// sg_kernels.cuh -- the day kernel, the external-transfer kernel and the
// recording helpers of the SimInf GB300 engine, templated on the model kind.
//
// Compiled twice: by nvcc into the library for the built-in kinds, and by
// NVRTC at run time for a model given as transition strings (the generated
// ModelTraits<SG_GENERIC> is defined before this header is included).  So it
// holds device code only and includes nothing but the engine's own headers.
#pragma once

#include "sg_common.h"
#include "sg_device.cuh"
#include "sg_filter.cuh"

namespace sg {

constexpr int kDayBlock = 128;
// Threads of the E2 kernel: the launch takes kE2Block when a replicate has more
// than kE2Small transfers a day (37,000 herds, 740 transfers a day: 14.7 ms a
// year with 256 threads, 13.3 with 512), else kE2Small (1,600 herds, 195 a
// day: 6.1 ms with either).
constexpr int kE2Block = 512, kE2Small = 256;

// Programmatic dependent launch: the day kernels and the E2 kernels are
// launched so that the next kernel in the stream may start while the
// previous one finishes.  Each kernel lets its successor launch at once,
// reads only static inputs (model tables, event plan) before pdl_wait, and
// waits for its predecessor (completion and memory) before it touches state.
// Every such kernel executes pdl_wait on all paths, so its completion implies
// its predecessor's.
__device__ __forceinline__ void pdl_trigger() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// ---------------------------------------------------------------------------
// Kernels
// ---------------------------------------------------------------------------

// Events of the plan in planned order (E1 part first).
struct EvDev {
  const SgEvent *rec;
  const int32_t *e1_day;       // day index of each E1 event
  const int64_t *e1_node_off;  // [slots * Nn + 1]; nullptr when there are none
};

__device__ __forceinline__ SgEvent load_event(const SgEvent *p) {
  union {
    int4 v[2];
    SgEvent e;
  } r;
  r.v[0] = __ldg(reinterpret_cast<const int4 *>(p));
  r.v[1] = __ldg(reinterpret_cast<const int4 *>(p) + 1);
  return r.e;
}

// Output selection (Sec. 3.2 result slots U_sparse and V_sparse, and the
// prevalence summary): compressed-column patterns with the layouts of U
// (rows node * C + compartment) and V (rows node * NV + index), one column
// per tspan point; values [R][nnz]; prevalence counters [R][M][4] (sum of
// cases, sum at risk, nodes with a case, nodes with anyone at risk).
struct OutDev {
  const int64_t *u_colptr = nullptr;
  const int32_t *u_row = nullptr;
  int32_t *u_val = nullptr;
  long long u_nnz = 0;
  const int64_t *v_colptr = nullptr;
  const int32_t *v_row = nullptr;
  double *v_val = nullptr;
  long long v_nnz = 0;
  uint32_t cases = 0, at_risk = 0;
  unsigned long long *prev = nullptr;
};

// First index in row[lo, hi) whose value is >= x.
__device__ __forceinline__ long long lower_bound_i32(const int32_t *row, long long lo,
                                                     long long hi, int32_t x) {
  while (lo < hi) {
    const long long mid = lo + ((hi - lo) >> 1);
    if (row[mid] < x) lo = mid + 1;
    else hi = mid;
  }
  return lo;
}

// The U_sparse / V_sparse entries of one node at tspan slot m.
template <int C, int NV>
__device__ __forceinline__ void record_sparse(const OutDev &o, int m, int rep, int node,
                                              const int *u, const double *v) {
  if (o.u_nnz > 0) {
    const long long hi = o.u_colptr[m + 1];
    long long e = lower_bound_i32(o.u_row, o.u_colptr[m], hi, node * C);
    for (; e < hi && o.u_row[e] < node * C + C; ++e) {
      const int p = o.u_row[e] - node * C;
      int x = 0;
#pragma unroll
      for (int q = 0; q < C; ++q)
        if (q == p) x = u[q];
      o.u_val[(long long)rep * o.u_nnz + e] = x;
    }
  }
  if (NV > 0 && o.v_nnz > 0) {
    const long long hi = o.v_colptr[m + 1];
    long long e = lower_bound_i32(o.v_row, o.v_colptr[m], hi, node * NV);
    for (; e < hi && o.v_row[e] < node * NV + NV; ++e) {
      const int p = o.v_row[e] - node * NV;
      double x = 0.0;
#pragma unroll
      for (int q = 0; q < NV; ++q)
        if (q == p) x = v[q];
      o.v_val[(long long)rep * o.v_nnz + e] = x;
    }
  }
}

// Adds recorded nodes to the prevalence counters of (replicate, slot m).
// Called by all 32 lanes of the warp together; `key` = rep * M + m for a
// thread that holds a unit (-1 otherwise; such lanes sit at the end of the
// warp, so equal keys are contiguous), `on` = its state is recorded.  A
// segmented inclusive scan over the warp, then one atomic per segment.
template <int C>
__device__ __forceinline__ void prevalence_add(const OutDev &o, long long key, bool on,
                                               const int *u) {
  long long cs = 0, rk = 0;
  int nc = 0, nr = 0;
  if (on) {
#pragma unroll
    for (int p = 0; p < C; ++p) {
      if ((o.cases >> p) & 1u) cs += u[p];
      if ((o.at_risk >> p) & 1u) rk += u[p];
    }
    nc = cs > 0;
    nr = rk > 0;
  }
  const unsigned full = 0xffffffffu;
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const long long k2 = __shfl_up_sync(full, key, d);
    const long long c2 = __shfl_up_sync(full, cs, d), r2 = __shfl_up_sync(full, rk, d);
    const int nc2 = __shfl_up_sync(full, nc, d), nr2 = __shfl_up_sync(full, nr, d);
    if (lane >= d && k2 == key) {
      cs += c2;
      rk += r2;
      nc += nc2;
      nr += nr2;
    }
  }
  const long long next = __shfl_down_sync(full, key, 1);
  if (key >= 0 && (lane == 31 || next != key)) {
    unsigned long long *q = o.prev + key * 4;
    if (cs) atomicAdd(q, (unsigned long long)cs);
    if (rk) atomicAdd(q + 1, (unsigned long long)rk);
    if (nc) atomicAdd(q + 2, (unsigned long long)nc);
    if (nr) atomicAdd(q + 3, (unsigned long long)nr);
  }
}

struct DayArgs {
  int *u;              // [R][Nn][C] working counts
  double *v;           // [R][Nn][NV] working continuous state
  const double *ldata; // [Nn][n_ldata]
  const int4 *ends;    // [Nn]: the season ends as integers (null: from ldata)
  int32_t *U;          // [R][M][Nn][C]
  double *V;           // [R][M][Nn][NV]
  const int32_t *rec;  // [days + 1]: tspan slot of T = t0 + i, or -1
  int32_t *e1_cur;     // [R][Nn]: next E1 event, relative to the node's list
  int32_t *e1_next;    // [R][Nn]: day index of that event, or SG_NO_DAY
  EvDev ev;
  int32_t t0, M, n_rep, slots;
  // global index of the run's replicate 0 (a shard of a larger job): every
  // random stream and error report uses rep0 + the local replicate, state
  // and outputs the local one
  int32_t rep0;
  // 1: the model's parameters are finite, so a unit without infected
  // animals and with phi == +0 has an empty day (k_days_sparse skips it)
  int32_t quiet;
  int32_t T_begin, T_end;  // SSA toward T = T_begin .. T_end - 1
  int32_t finish_first;    // finish unit step T_begin - 1 before the SSA
  int32_t finish_last;     // finish unit step T_end - 1 after the SSA
  int32_t heavy_after;     // aem, or intervals that do not apply: draws a thread
                           // takes before a warp takes over
  // the intervals of sg_filter.cuh apply: parameters finite and not negative,
  // every rate a function of the counts (G marks at least the rates that each
  // transition changes), and S the kind's own (1) or a caller's (2); 0: not
  int32_t fast;
  float warp_rate;         // expected transitions from which a unit's day goes to a warp,
  int32_t warp_max;        // if the block has at most this many such units
  int32_t npb;             // nodes per block (<= kDayBlock); the other
                           // threads of the block only serve heavy nodes
  const int32_t *emu;      // [R][Nn][4]: emulated increments of I_1..I_3 and
                           // a flag (1 = use them instead of the SSA), or null
  // the emulator's node split across two launches of a day: 0 every node;
  // 1 only the nodes outside the emulator's range (emu_flag[gid] == 0, the
  // SSA part, run beside the emulator); 2 only the emulated nodes (emu[gid]
  // flag set)
  const int32_t *emu_flag;
  int32_t emu_part;
  uint32_t k0, k1;         // Philox key (seed)
  SgDevError *err;
  SgCounters *cnt;
  // all events method: channel state [T][R * Nn] (rate, firing time, draws
  // taken); null for the direct method
  double *aem_a, *aem_tau;
  uint32_t *aem_cnt;
  OutDev out;            // sparse output and prevalence (U, V may be null)
  // external transfers of unit time T_end - 1 run inside this launch, by the
  // last block to finish each replicate's nodes (null: none or by the E2
  // kernel): wave bounds (wave_ev), the day's wave range [e2_wb, e2_we) when
  // the events are shared, else per replicate from wave_off[day][slot], and
  // a per-replicate count of finished blocks (zero between launches)
  const int64_t *wave_ev, *wave_off;
  long long e2_wb, e2_we;
  int32_t e2_day_index;
  int32_t *e2_done;
  // persistent run (cooperative launch, every block resident): the days'
  // external transfers run inside this launch between two grid barriers
  // (arrival count, generation); null: not persistent
  unsigned int *grid_bar;
  int32_t n_blocks;
  // sparse schedule with every block holding whole replicates (nodes per
  // block a multiple of the node count): each block runs its replicates'
  // external transfers of every day itself, between the day's E1 events and
  // its post time step, so one launch covers all days; 0: off
  int32_t e2_inblock;
};

// A node's season ends as integers (the conversion from ldata is a dozen FP64
// instructions, so it is done once per model).
__device__ __forceinline__ void load_ends(const int4 *ends, const double *ldata,
                                          const SgTables &tb, int node, int *ld) {
  if (ends) {
    const int4 e = __ldg(ends + node);
    ld[0] = e.x;
    ld[1] = e.y;
    ld[2] = e.z;
    ld[3] = e.w;
  } else {
#pragma unroll
    for (int i = 0; i < 4; ++i) ld[i] = season_end_int(ldata[(long long)node * tb.n_ldata + i]);
  }
}

// %globaltimer (ns).
__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// Adds one recorded unit to the prevalence counters of `key` with its own
// atomics (for units taken from a list, whose lanes are in no order).
template <int C>
__device__ __forceinline__ void prevalence_add_unit(const OutDev &o, long long key,
                                                    const int *u) {
  long long cs = 0, rk = 0;
#pragma unroll
  for (int p = 0; p < C; ++p) {
    if ((o.cases >> p) & 1u) cs += u[p];
    if ((o.at_risk >> p) & 1u) rk += u[p];
  }
  unsigned long long *q = o.prev + key * 4;
  if (cs) atomicAdd(q, (unsigned long long)cs);
  if (rk) atomicAdd(q + 1, (unsigned long long)rk);
  if (cs > 0) atomicAdd(q + 2, 1ull);
  if (rk > 0) atomicAdd(q + 3, 1ull);
}

// A grid barrier must wait for the slowest block's whole day; a wait longer
// than this is taken as a failure (SG_ERR_TIMEOUT) instead of a hang.
constexpr unsigned long long kGridWaitNs = 20ull * 1000 * 1000 * 1000;

// Grid-wide barrier for a cooperative launch (all blocks resident): thread 0
// of each block reads the generation, fences, arrives; the last arrival
// resets the count and advances the generation; the others poll the
// generation with a time limit.  Returns false (the same in every thread of
// the block) if this block gave up; the kernel must then leave.
__device__ __forceinline__ bool grid_barrier(unsigned int *bar, int n_blocks, SgDevError *err) {
  __shared__ int s_ok;
  __syncthreads();
  if (threadIdx.x == 0) {
    volatile unsigned int *gen = bar + 1;
    const unsigned int g = *gen;
    __threadfence();
    int ok = 1;
    if (atomicAdd(bar, 1u) == (unsigned int)n_blocks - 1u) {
      atomicExch(bar, 0u);
      __threadfence();
      atomicAdd(bar + 1, 1u);
    } else {
      const unsigned long long t0 = global_ns();
      while (*gen == g) {
        if (global_ns() - t0 > kGridWaitNs) {
          ok = 0;
          report(err, SG_ERR_TIMEOUT, -1, -1, -1, -1);
          break;
        }
        __nanosleep(100);
      }
    }
    __threadfence();
    s_ok = ok;
  }
  __syncthreads();
  return s_ok != 0;
}

// A day's events and wave bounds staged in shared memory while the day's SSA
// runs, for e2_rep_block.
constexpr int kE2StageEv = 128, kE2StageWaves = 31;
struct E2Stage {
  SgEvent ev[kE2StageEv];
  long long wave[kE2StageWaves + 1];  // bounds of waves w0 .. w0 + n_waves
  long long w0, w1, lo;               // the day's waves, first staged event
  int n_waves, n_ev;                  // 0: nothing staged
};

// Staged by one warp, the events by asynchronous copies that the block waits
// for (cp.async.wait_all and a barrier) before e2_rep_block.
__device__ __forceinline__ void e2_stage(E2Stage &s, const DayArgs &a, long long w0,
                                         long long w1) {
  const int lane = threadIdx.x & 31;
  const int nw = (int)min(w1 - w0, (long long)kE2StageWaves);
  if (lane <= nw) s.wave[lane] = a.wave_ev[w0 + lane];
  __syncwarp();
  const long long lo = s.wave[0];
  const int n = (int)min(s.wave[nw] - lo, (long long)kE2StageEv);
  if (lane == 0) {
    s.w0 = w0;
    s.w1 = w1;
    s.lo = lo;
    s.n_waves = nw;
    s.n_ev = n;
  }
  for (int i = lane; i < 2 * n; i += 32)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                     (uint32_t)__cvta_generic_to_shared(reinterpret_cast<int4 *>(s.ev) + i)),
                 "l"(reinterpret_cast<const int4 *>(a.ev.rec + lo) + i)
                 : "memory");
}

// The number of large transfers that a wave left to the warps (the same in
// every thread), read after the wave's barrier; three counters take turns.  A
// fast thread may add to the next wave's counter before a slow one has read
// this wave's, so they differ; the one cleared here was last read before this
// wave's barrier and is added to after the next one's.
__device__ __forceinline__ int next_wave(int *count, int &cw) {
  const int n = count[cw];
  if (threadIdx.x == 0) count[cw == 0 ? 2 : cw - 1] = 0;
  cw = cw == 2 ? 0 : cw + 1;
  return n;
}

// The external transfers (Sec. 3.3) of replicate `rep` at unit time T, wave by
// wave, by one block (a block barrier between waves), on the replicate's
// state in global memory.  The state was written by other blocks of the same
// launch, so it is read and written at L2 only (ld / st .cg) and added to
// with atomics; a wave never samples a node another event of the wave
// touches.  Same arithmetic and random stream as the E2 kernel.  Returns
// whether a transfer failed (the same in every thread).
template <int C>
__device__ bool e2_rep_block(const SgTables &tb, const DayArgs &a, int rep, int T,
                             long long w0, long long w1, const E2Stage *stage = nullptr) {
  auto event = [&](long long j) {
    if (stage && j >= stage->lo && j < stage->lo + stage->n_ev) return stage->ev[j - stage->lo];
    return load_event(a.ev.rec + j);
  };
  auto bound = [&](long long w) {
    if (stage && w >= stage->w0 && w <= stage->w0 + stage->n_waves)
      return stage->wave[w - stage->w0];
    return (long long)a.wave_ev[w];
  };
  // a run that already failed does nothing (one thread reads, the barrier
  // makes the answer the block's); with the events staged the caller knows
  // whether its own units' day went well
  if (!stage && __syncthreads_or(threadIdx.x == 0 && *(volatile int32_t *)&a.err->code != 0))
    return true;
  int *state = a.u + (long long)rep * tb.n_nodes * C;
  const uint64_t seed = ((uint64_t)a.k1 << 32) | a.k0;
  constexpr int kHv = 256;  // large transfers of a wave left to the warps
  __shared__ long long s_hv[kHv];
  __shared__ int s_nhv[3];  // see next_wave
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
  unsigned long long applied = 0;
  bool bad = false, failed = false;
  if (threadIdx.x < 3) s_nhv[threadIdx.x] = 0;
  int cw = 0;
  __syncthreads();
  for (long long w = w0; w < w1; ++w) {
    const long long lo = bound(w), hi = bound(w + 1);
    for (long long j = lo + threadIdx.x; j < hi; j += blockDim.x) {
      const SgEvent ev = event(j);
      const int src = ev.node;
      int *un = state + (long long)src * C;
      const uint32_t mask = tb.Emask[ev.select];
      const long long idx = ev.index;
      int cur[C];
      long long total = 0;
#pragma unroll
      for (int p = 0; p < C; ++p) {
        cur[p] = __ldcg(un + p);
        if ((mask >> p) & 1u) total += cur[p];
      }
      const long long k =
          ev.n > 0 ? (long long)ev.n : (long long)round(ev.proportion * (double)total);
      if (k < 0 || k > total) {
        report(a.err, SG_ERR_EVENT_UNDERFLOW, a.rep0 + rep, src, T, idx);
        bad = true;
        continue;
      }
      if (k >= kUrnWarp) {
        // a large transfer: sampled by a warp after this pass (in this
        // thread when the list is full)
        const int slot = atomicAdd(&s_nhv[cw], 1);
        if (slot < kHv) {
          s_hv[slot] = j;
          continue;
        }
      }
      int moved[C];
#pragma unroll
      for (int p = 0; p < C; ++p) moved[p] = 0;
      if (k > 0) {
        WordStream ws;
        ws.init(seed, idx, a.rep0 + rep);
        for (long long d = 0; d < k; ++d) {
          uint32_t x = ws.below((uint32_t)(total - d));
          bool taken = false;
#pragma unroll
          for (int p = 0; p < C; ++p) {
            if (taken || !((mask >> p) & 1u)) continue;
            const uint32_t rem = (uint32_t)(cur[p] - moved[p]);
            if (x < rem) {
              ++moved[p];
              taken = true;
            } else {
              x -= rem;
            }
          }
        }
      }
      const int q_sh = ev.shift;
      int *ud = state + (long long)ev.dest * C;
#pragma unroll
      for (int p = 0; p < C; ++p)
        if (moved[p] != 0) __stcg(un + p, cur[p] - moved[p]);
#pragma unroll
      for (int p = 0; p < C; ++p)
        if (moved[p] != 0) atomicAdd(ud + (q_sh >= 0 ? p + tb.Nsh[q_sh][p] : p), moved[p]);
      ++applied;
    }
    // one barrier per wave; its result is the same for every thread
    if (__syncthreads_or(bad)) {
      failed = true;
      break;
    }
    const int nhv = min(next_wave(s_nhv, cw), kHv);
    if (nhv > 0) {
      // the wave's large transfers, one warp each (no other event of the
      // wave touches their source nodes)
      for (int h = warp; h < nhv; h += nwarps) {
        const long long j = s_hv[h];
        const SgEvent ev = event(j);
        const int src = ev.node;
        int *un = state + (long long)src * C;
        const uint32_t mask = tb.Emask[ev.select];
        int cur[C];
        long long total = 0;
#pragma unroll
        for (int p = 0; p < C; ++p) {
          cur[p] = __ldcg(un + p);
          if ((mask >> p) & 1u) total += cur[p];
        }
        const long long k =
            ev.n > 0 ? (long long)ev.n : (long long)round(ev.proportion * (double)total);
        int moved[C];
        urn_warp<C>(cur, mask, (uint32_t)k, (uint32_t)total, seed, ev.index, a.rep0 + rep,
                    moved);
        if (lane == 0) {
          const int q_sh = ev.shift;
          int *ud = state + (long long)ev.dest * C;
#pragma unroll
          for (int p = 0; p < C; ++p)
            if (moved[p] != 0) __stcg(un + p, cur[p] - moved[p]);
#pragma unroll
          for (int p = 0; p < C; ++p)
            if (moved[p] != 0) atomicAdd(ud + (q_sh >= 0 ? p + tb.Nsh[q_sh][p] : p), moved[p]);
          ++applied;
        }
        __syncwarp();
      }
      __syncthreads();
    }
  }
  if (applied) atomicAdd(&a.cnt->events, applied);
  return failed;
}

// u += S[, n] and the rates that column n of G marks recomputed; 0 or
// SG_ERR_RATE.
template <int KIND>
__device__ __forceinline__ int apply_transition(int *u, double *w, int n, const double *kf,
                                                const SgTables &tb) {
  using M = ModelTraits<KIND>;
#pragma unroll
  for (int p = 0; p < M::C; ++p) u[p] += tb.S[n][p];
  const uint32_t dep = tb.dep[n];
  int code = 0;
#pragma unroll
  for (int k = 0; k < M::T; ++k) {
    if ((dep >> k) & 1u) {
      w[k] = M::rate_k(k, u, kf, tb.gdata);
      if (bad_rate(w[k])) code = SG_ERR_RATE;
    }
  }
  return code;
}

// One transition (Appendix A, inversion and update): the smallest n with
// target <= running sum of the positive rates (last positive one if rounding
// leaves none), then apply_transition.
template <int KIND>
__device__ __forceinline__ int fire(int *u, double *w, double target, const double *kf,
                                    const SgTables &tb) {
  using M = ModelTraits<KIND>;
  // running sum over the positive rates in index order; the first term is
  // taken as is (0 + w == w exactly), the comparisons are exact integer
  // comparisons of non-negative doubles
  double cum = 0.0;
  int n = -1, last = -1;
#pragma unroll
  for (int j = 0; j < M::T; ++j) {
    if (n < 0 && gt0(w[j])) {
      cum = last < 0 ? w[j] : cum + w[j];
      last = j;
      if (le_nonneg(target, cum)) n = j;
    }
  }
  if (n < 0) n = last;
  return apply_transition<KIND>(u, w, n, kf, tb);
}

// Prefix sums P_j = (..(w_0 + w_1) + ..) + w_j of the rates in index order.
// P_(T-1) is lambda as the direct method sums it, and at every positive rate P_j is
// the running sum of the positive rates that fire() forms (adding a zero
// rate leaves a sum unchanged, and a sum of zeros plus w is w).
template <int T>
__device__ __forceinline__ void rate_prefix(const double *w, double *P) {
#pragma unroll
  for (int j = 0; j < T; ++j) P[j] = j == 0 ? w[0] : P[j - 1] + w[j];
}

// fire()'s choice of transition from the prefix sums.
template <int T>
__device__ __forceinline__ int select_prefix(const double *w, const double *P, double target) {
  int n = -1, last = -1;
#pragma unroll
  for (int j = 0; j < T; ++j) {
    if (gt0(w[j])) {
      if (n < 0) last = j;
      if (n < 0 && le_nonneg(target, P[j])) n = j;
    }
  }
  return n < 0 ? last : n;
}

enum { SSA_DONE = 0, SSA_REDO = 1 };

// Direct SSA of one unit's day toward Td in its own thread, every operation
// in FP64 (Appendix A, one iteration per draw).  Returns SSA_DONE, SSA_REDO
// (counts unchanged: more than `budget` draws were due, the day is left to a
// warp, which starts it again because rates kept by a caller's own G depend
// on the way to a state) or an error.
template <int KIND>
__device__ __forceinline__ int ssa_exact(int *u0, const double *kf, uint32_t node, uint32_t Td,
                                         uint32_t tag, uint32_t k0, uint32_t k1, int budget,
                                         const SgTables &tb, unsigned long long &fired,
                                         unsigned long long &drawn) {
  using M = ModelTraits<KIND>;
  const double Tn = (double)(int)Td;
  const long long Tkey = order_key(Tn);
  double t = (double)((int)Td - 1);
  uint32_t c = 0, f = 0;
  int code = SSA_DONE;
  int u[M::C];
  double w[M::T];
#pragma unroll
  for (int p = 0; p < M::C; ++p) u[p] = u0[p];
#pragma unroll
  for (int j = 0; j < M::T; ++j) {
    w[j] = M::rate_k(j, u, kf, tb.gdata);
    if (bad_rate(w[j])) code = SG_ERR_RATE;
  }
  while (code == SSA_DONE) {
    // lambda = ((0 + w_1) + w_2) + ...; the leading 0 + w_1 changes no
    // decision or value, so the sum starts at w_1
    double lam = w[0];
#pragma unroll
    for (int j = 1; j < M::T; ++j) lam = lam + w[j];
    if (!gt0(lam)) break;  // nothing can fire: jump to Tn
    if (c >= SG_MAX_DRAWS) {
      code = SG_ERR_STEP_LIMIT;
      break;
    }
    if (c == (uint32_t)budget) return SSA_REDO;
    const U4 x = philox10(U4{c, node, Td, tag}, k0, k1);
    ++c;
    const double tau = -log_pos(u01_open(x.x, x.y)) / lam;
    const double tt = t + tau;
    if (order_key(tt) >= Tkey) break;
    t = tt;
    code = fire<KIND>(u, w, lam * u01_open(x.z, x.w), kf, tb);
    ++f;
  }
#pragma unroll
  for (int p = 0; p < M::C; ++p) u0[p] = u[p];
  fired += f;
  drawn += c;
  return code;
}

// A unit's day left to a warp, from its start.
template <int C, int NK>
struct HeavySlot {
  double kf[NK];
  int32_t node, rep, code;
  int32_t redo;  // 1: intervals have left the day's end open in its thread
  int32_t u[C];
};

// The transition that lambda r2 selects with the rates of the counts u in
// FP64 (the intervals of sg_filter.cuh did not settle it): -1 if no rate is
// positive.  w2, w3: the draw's third and fourth Philox words.
template <int KIND>
__device__ __forceinline__ int select_exact(const int *u, const double *kf, uint32_t w2,
                                            uint32_t w3, const SgTables &tb) {
  using M = ModelTraits<KIND>;
  double w[M::T], P[M::T];
#pragma unroll
  for (int j = 0; j < M::T; ++j) w[j] = M::rate_k(j, u, kf, tb.gdata);
  rate_prefix<M::T>(w, P);
  if (!gt0(P[M::T - 1])) return -1;
  return select_prefix<M::T>(w, P, P[M::T - 1] * u01_open(w2, w3));
}

// Time since the day's start, an interval [lo, hi] in units of 2^-31 of the
// day, its ends rounded outward and each waiting time cut at one day (so the
// sums stay below 2^32).  FP64's own rounding of t + tau moves the time by at
// most half an ulp at |T| + 1 per transition, (|T| + 1) 2^-22 units; drift
// is that in 2^-6 units, rounded up, and d the number of transitions
// (at most kFilterDraws, so d * drift < 2^32).
constexpr uint32_t kDayUnits = 1u << 31;
// Longer days take exact times at once: with n draws the end of the day is left
// open in n (2.5e-6 + n 5e-10) of the cases, and the attempt is lost.
constexpr uint32_t kFilterDraws = 1u << 15;
struct DayTime {
  uint32_t lo = 0, hi = 0, d = 0, drift;
  __device__ __forceinline__ explicit DayTime(uint32_t Td)
      : drift((((uint32_t)abs((int)Td) + 1u) >> 16) + 1u) {}
  __device__ __forceinline__ void add(uint32_t t_lo, uint32_t t_hi) {
    lo += t_lo;
    hi += t_hi;
    ++d;
  }
  // t + tau >= Tn certainly
  __device__ __forceinline__ bool after(uint32_t t_lo) const {
    return lo + t_lo >= kDayUnits + ((d * drift + 63u) >> 6);
  }
  // t + tau < Tn certainly for each of the next n draws, which take at most
  // t_hi together
  __device__ __forceinline__ bool before(uint32_t t_hi, uint32_t n) const {
    return hi + t_hi < kDayUnits - (((d + n) * drift + 63u) >> 6);
  }
};
__device__ __forceinline__ uint32_t day_units_lo(float t) {
  return __float2uint_rd(fminf(t, 1.0f) * 0x1.0p31f);
}
__device__ __forceinline__ uint32_t day_units_hi(float t) {
  return __float2uint_ru(fminf(t, 1.0f) * 0x1.0p31f);
}

// Direct SSA of one unit's whole day in its thread, decided from intervals
// (sg_filter.cuh): same draws, same transitions and same end as ssa_exact.
// Returns SSA_DONE with the counts after the day in u, or SSA_REDO (counts
// unchanged) where an interval does not settle the time of
// an event or applies no more: the day must then run with exact times.
//
// Cost: a draw is ~150 instructions, none of them FP64 (the FP64 form of it
// is 55 FP64 instructions of ~76 issue cycles each).  The random numbers of
// the next draw do not depend on this one's outcome, so they are computed
// beside it.  Bound by issue where every lane has a unit (100,000 endemic
// SISe3 herds x 20 days, 130 M draws: 3.2 ms, in FP64 43.0 ms), elsewhere by
// the latency of the longest unit (100 SIR nodes x 99 days: 0.19 ms, 1.33 ms).
template <int KIND, typename F_t = Filter<KIND>>
__device__ __forceinline__ int ssa_filter(int *u, const double *kf, uint32_t node, uint32_t Td,
                                          uint32_t tag, uint32_t k0, uint32_t k1,
                                          const SgTables &tb, unsigned long long &fired,
                                          unsigned long long &drawn) {
  using M = ModelTraits<KIND>;
  constexpr int T = M::T;
  F_t F;
  if (!F.load(u, kf, tb)) return SSA_REDO;
  DayTime t(Td);
  U4 x = philox10(U4{0u, node, Td, tag}, k0, k1);
  Itv E = itv_neglog(x.x, x.y);
  for (;;) {
    const U4 xn = philox10(U4{t.d + 1u, node, Td, tag}, k0, k1);
    const Itv En = itv_neglog(xn.x, xn.y);
    Itv P[T];
    const bool good = F.sums(P, tb);
    const float l_lo = P[T - 1].lo, l_hi = P[T - 1].hi;
    if (good && l_hi == 0.0f) {  // nothing can fire: jump to Tn
      drawn += t.d;
      break;
    }
    if (!(good && l_lo >= kItvMin && l_hi <= kItvMax) || t.d >= kFilterDraws)
      return SSA_REDO;
    // tau = E / lambda
    const uint32_t t_lo = day_units_lo(__fmul_rd(E.lo, rcp_lo(l_hi)));
    const uint32_t t_hi = day_units_hi(__fmul_ru(E.hi, rcp_hi(l_lo)));
    if (t.after(t_lo)) {  // the draw is discarded
      drawn += t.d + 1u;
      break;
    }
    if (!t.before(t_hi, 1)) return SSA_REDO;
    t.add(t_lo, t_hi);
    int n = itv_select<T>(P, itv_r2(x.w));
    if (n < 0) {
      int v[M::C];
#pragma unroll
      for (int p = 0; p < M::C; ++p) v[p] = (int)F.x[p];
      n = select_exact<KIND>(v, kf, x.z, x.w, tb);
      if (n < 0) return SSA_REDO;
    }
    F.fire(n, tb);
    x = xn;
    E = En;
  }
#pragma unroll
  for (int p = 0; p < M::C; ++p) u[p] = (int)F.x[p];
  fired += t.d;  // every draw but the one that passed Tn
  return SSA_DONE;
}

// One unit's day in its thread where the kind's own intervals do not apply, by
// FilterWide (own: a caller's own S) or with exact times.  Out of line, so that
// k_days keeps its registers for ssa_filter.  u and kf are copies that the
// caller makes for this call; n[0] and n[1] get the day's transitions and draws.
template <int KIND>
__device__ __noinline__ int ssa_general(int *u, const double *kf, uint32_t node, uint32_t Td,
                                        uint32_t tag, uint32_t k0, uint32_t k1, bool own,
                                        int budget, const SgTables &tb, unsigned long long *n) {
  unsigned long long f = 0, d = 0;
  const int r = own ? ssa_filter<KIND, FilterWide<KIND>>(u, kf, node, Td, tag, k0, k1, tb, f, d)
                    : ssa_exact<KIND>(u, kf, node, Td, tag, k0, k1, budget, tb, f, d);
  n[0] = f;
  n[1] = d;
  return r;
}

// One unit's day in its thread, by what `fast` says (DayArgs::fast).
template <int KIND>
__device__ __forceinline__ int ssa_thread(int *u, const double *kf, uint32_t node, uint32_t Td,
                                          uint32_t tag, uint32_t k0, uint32_t k1, int fast,
                                          int budget, const SgTables &tb,
                                          unsigned long long &fired, unsigned long long &drawn) {
  using M = ModelTraits<KIND>;
  // a model from transition strings is always 1
  if (KIND == SG_GENERIC || fast == 1)
    return ssa_filter<KIND>(u, kf, node, Td, tag, k0, k1, tb, fired, drawn);
  int un[M::C];
  double kn[M::NK];
  unsigned long long n[2];
#pragma unroll
  for (int p = 0; p < M::C; ++p) un[p] = u[p];
#pragma unroll
  for (int i = 0; i < M::NK; ++i) kn[i] = kf[i];
  const int r = ssa_general<KIND>(un, kn, node, Td, tag, k0, k1, fast == 2, budget, tb, n);
#pragma unroll
  for (int p = 0; p < M::C; ++p) u[p] = un[p];
  fired += n[0];
  drawn += n[1];
  return r;
}

// The day's total rate as an interval; false (lambda not set) where the intervals
// do not apply.
template <int KIND>
__device__ __forceinline__ bool day_rate(const int *u, const double *kf, int fast,
                                         const SgTables &tb, Itv &lambda) {
  constexpr int T = ModelTraits<KIND>::T;
  Itv L[T];
  bool good = false;
  if (KIND == SG_GENERIC || fast == 1) {
    Filter<KIND> F;
    good = F.load(u, kf, tb) && F.sums(L, tb);
  } else if (fast == 2) {
    FilterWide<KIND> F;
    good = F.load(u, kf, tb) && F.sums(L, tb);
  }
  if (good) lambda = L[T - 1];
  return good;
}

// Direct SSA of one unit's day by a whole warp, decided from intervals.  The
// draws depend only on (seed, replicate, node, day, draw index), so lane l
// holds the random numbers of draw c0 + l.  The states that the next J draws
// can reach are the counts plus a multiset of at most J - 1 transitions; each
// lane evaluates one of them at its draw (running sums, waiting time,
// transition), and the walk then follows the fired transitions through the
// lanes.  One or two transitions: J = 8, 7 and lane j (j + 1) / 2 + b (b
// times the second one after j); three to six: J = 3, lanes in order of the
// root, single transitions and sorted pairs; more: J = 2.
//
// Latency bound: a round is one evaluation and J dependent shuffles.  At ten
// times a thread's instructions it pays for the few units of a block whose
// day is long (1,000 predator-prey nodes x 30 days, 2,600 draws a node-day:
// 15.8 ms, by threads 38.7 ms; 37,000 SISe3 herds x 365 days: 13.3 ms, 17.1
// ms).
template <int T>
struct Window {
  static constexpr int J = T == 1 ? 8 : T == 2 ? 7 : T <= 6 ? 3 : 2;
};
template <int KIND, typename F_t>
__device__ __forceinline__ int ssa_window(int *u, const double *kf, uint32_t node, uint32_t Td,
                                          uint32_t tag, uint32_t k0, uint32_t k1,
                                          const SgTables &tb, unsigned long long &fired,
                                          unsigned long long &drawn) {
  using M = ModelTraits<KIND>;
  constexpr int C = M::C, T = M::T, J = Window<T>::J;
  constexpr unsigned full = 0xffffffffu;
  constexpr int kNone = T, kOpen = T + 1, kBad = T + 2;  // no transition; not settled; no interval
  const int lane = threadIdx.x & 31;
  F_t F;
  if (!F.load(u, kf, tb)) return SSA_REDO;
  {
    Itv L[T];
    if (F.sums(L, tb) && L[T - 1].lo >= (float)kFilterDraws) return SSA_REDO;
  }
  // this lane's multiset: its size and what it adds to the counts
  int depth = 0;
  decltype(F.x[0] + F.x[0]) add[C];
  {
    int m0 = -1, m1 = -1, n0 = 0, n1 = 0;  // n0 times m0 and n1 times m1
    if (T <= 2) {
      int l = lane < (T == 1 ? J : J * (J + 1) / 2) ? lane : 0;
      if (T == 1) {
        depth = n0 = l;
      } else {
        while (l > depth) l -= ++depth;
        n1 = l;
        n0 = depth - l;
      }
      m0 = 0;
      m1 = T - 1;
    } else if (lane >= 1 && lane <= T) {
      depth = n0 = 1;
      m0 = lane - 1;
    } else if (J == 3 && lane > T && lane < 1 + T + T * (T + 1) / 2) {
      depth = 2;
      n0 = n1 = 1;
      int l = lane - 1 - T;
      m0 = 0;
      while (l >= T - m0) l -= T - m0++;
      m1 = m0 + l;
    }
#pragma unroll
    for (int p = 0; p < C; ++p) {
      int y = 0;
      if (m0 >= 0 && n0) y += n0 * tb.S[m0][p];
      if (m1 >= 0 && n1) y += n1 * tb.S[m1][p];
      add[p] = y;
    }
  }
  DayTime t(Td);
  uint32_t c0 = 0, w2 = 0, w3 = 0;
  float e_lo = 0.0f, e_hi = 0.0f;
  bool have = false;
  for (;;) {
    if (!have || t.d + (uint32_t)J - c0 > 32u) {
      if (t.d >= kFilterDraws) return SSA_REDO;
      c0 = t.d;
      const U4 x = philox10(U4{c0 + (uint32_t)lane, node, Td, tag}, k0, k1);
      const Itv E = itv_neglog(x.x, x.y);
      e_lo = E.lo;
      e_hi = E.hi;
      w2 = x.z;
      w3 = x.w;
      have = true;
    }
    F_t G = F;
#pragma unroll
    for (int p = 0; p < C; ++p) G.x[p] += add[p];
    const int src = (int)(t.d - c0) + depth;
    const float El = __shfl_sync(full, e_lo, src), Eh = __shfl_sync(full, e_hi, src);
    const uint32_t r = __shfl_sync(full, w3, src);
    Itv P[T];
    const bool good = G.sums(P, tb);
    const float l_lo = P[T - 1].lo, l_hi = P[T - 1].hi;
    // the waiting time
    const uint32_t t_lo = day_units_lo(__fmul_rd(El, rcp_lo(l_hi)));
    const uint32_t t_hi = day_units_hi(__fmul_ru(Eh, rcp_hi(l_lo)));
    int n = itv_select<T>(P, itv_r2(r));
    if (n < 0) n = kOpen;
    if (!(good && l_lo >= kItvMin && l_hi <= kItvMax)) n = good && l_hi == 0.0f ? kNone : kBad;
    // the lanes of the states on the way, and what their draws add up to
    int m[J], L = 0, b = 0;
    uint32_t a_lo[J], a_hi[J], sum_hi = 0;
    bool all = true;
#pragma unroll
    for (int j = 0; j < J; ++j) {
      m[j] = __shfl_sync(full, n, L);
      a_lo[j] = __shfl_sync(full, t_lo, L);
      a_hi[j] = __shfl_sync(full, t_hi, L);
      all = all && m[j] < kNone;
      if (T <= 2) {
        b += T == 2 ? m[j] : 0;
        L = T == 1 ? j + 1 : ((j + 1) * (j + 2) / 2 + b) & 31;
      } else if (j == 0) {
        L = (1 + m[0]) & 31;
      } else if (j == 1) {
        const int lo = min(m[0], m[1]), hi = max(m[0], m[1]);
        L = (1 + T + lo * T - lo * (lo - 1) / 2 + (hi - lo)) & 31;
      }
      sum_hi = min(sum_hi + a_hi[j], kDayUnits - 1u);
    }
    if (all && t.before(sum_hi, J)) {  // every one of them falls into the day
#pragma unroll
      for (int j = 0; j < J; ++j) {
        t.add(a_lo[j], a_hi[j]);
        F.fire(m[j], tb);
      }
      continue;
    }
    // otherwise one draw at a time; after a draw that the intervals do not
    // settle, a new round
#pragma unroll
    for (int j = 0; j < J; ++j) {
      if (m[j] == kBad) return SSA_REDO;
      if (m[j] == kNone || t.after(a_lo[j])) {
        drawn += m[j] == kNone ? t.d : t.d + 1u;
        fired += t.d;
#pragma unroll
        for (int p = 0; p < C; ++p) u[p] = (int)F.x[p];
        return SSA_DONE;
      }
      if (!t.before(a_hi[j], 1)) return SSA_REDO;
      const bool open = m[j] == kOpen;
      if (open) {
        int v[C];
#pragma unroll
        for (int p = 0; p < C; ++p) v[p] = (int)F.x[p];
        const uint32_t x2 = __shfl_sync(full, w2, (int)(t.d - c0));
        const uint32_t x3 = __shfl_sync(full, w3, (int)(t.d - c0));
        m[j] = select_exact<KIND>(v, kf, x2, x3, tb);
        if (m[j] < 0) return SSA_REDO;
      }
      t.add(a_lo[j], a_hi[j]);
      F.fire(m[j], tb);
      if (open) break;
    }
  }
}

// The transitions of up to 32 draws from the counts in F on, each selected
// from intervals or in FP64: lane l of `us` gets the counts before draw l,
// F.x the ones after the last walked draw.  x: lane l's Philox words of draw
// l, e_lo its waiting time's lower end, left: what is left of the day, rounded
// up.  Returns whether a state after the last walked draw exists (not where
// nothing can fire, or the day is surely over).
template <int KIND, typename F_t>
__device__ __forceinline__ bool walk_draws(F_t &F, const U4 &x, float e_lo, float left,
                                           const double *kf, const SgTables &tb, int *us,
                                           int &walked) {
  using M = ModelTraits<KIND>;
  constexpr int C = M::C, T = M::T;
  constexpr unsigned full = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  for (walked = 0; walked < 32;) {
    Itv P[T];
    const bool good = F.sums(P, tb) && P[T - 1].lo >= kItvMin && P[T - 1].hi <= kItvMax;
    const uint32_t w2 = __shfl_sync(full, x.z, walked), w3 = __shfl_sync(full, x.w, walked);
    const float e = __shfl_sync(full, e_lo, walked);
    int v[C];
#pragma unroll
    for (int p = 0; p < C; ++p) v[p] = (int)F.x[p];
    if (lane == walked) {
#pragma unroll
      for (int p = 0; p < C; ++p) us[p] = v[p];
    }
    ++walked;
    int n = good ? itv_select<T>(P, itv_r2(w3)) : -1;
    if (n < 0) n = select_exact<KIND>(v, kf, w2, w3, tb);
    if (good) left -= e * rcp_lo(P[T - 1].hi);
    if (n < 0 || left < 0.0f) return false;
    F.fire(n, tb);
  }
  return true;
}

// Direct SSA of one unit by a whole warp: from intervals (ssa_window), and
// where they leave an event's time open, with exact times.
//
// With the kind's own tables (`fast`): the transitions of up to 32 draws are
// walked first, selected from intervals (they depend on the draws' r2 and
// the counts, not on the times), and lane l keeps the counts before draw l
// (a day may take them anywhere in int32: FP32 counts are loaded anew for
// every 32 draws, and where they would not be exact FilterWide takes over);
// then every lane evaluates its draw in FP64 -- rates, lambda and E / lambda,
// 32 logarithms and divisions for the price of one -- and the times are
// added up in order, which tells where the day ends.  A draw walked beyond
// that is dropped.  Same values as one draw after the other, since the rates
// are functions of the counts.
//
// Otherwise (a caller's own S or G): draw by draw, the rates kept as G says;
// the lanes only compute 32 draws' random numbers at once.
template <int KIND>
__device__ __noinline__ void ssa_warp(
    HeavySlot<ModelTraits<KIND>::C, ModelTraits<KIND>::NK> &hs, double Tn, uint32_t Td,
    uint32_t k0, uint32_t k1, int fast, const SgTables &tb, unsigned long long &fired,
    unsigned long long &drawn) {
  using M = ModelTraits<KIND>;
  constexpr int C = M::C, T = M::T, NK = M::NK;
  constexpr unsigned full = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  int u[C];
  double kf[NK];
#pragma unroll
  for (int p = 0; p < C; ++p) u[p] = hs.u[p];
#pragma unroll
  for (int i = 0; i < NK; ++i) kf[i] = hs.kf[i];
  double t = Tn - 1.0;
  uint32_t c = 0;
  const uint32_t node = (uint32_t)hs.node;
  const uint32_t tag = (SG_STREAM_SSA << 24) | (uint32_t)hs.rep;
  int code = 0;
  unsigned long long f = 0, wf = 0, wd = 0;
  const long long Tkey = order_key(Tn);
  int r = SSA_REDO;
  if (fast) {
    // (a thread that gave up has decided from the same intervals)
    Filter<KIND> N;
    if (fast == 1 && N.load(u, kf, tb)) {
      if (!hs.redo)
        r = ssa_window<KIND, Filter<KIND>>(u, kf, node, Td, tag, k0, k1, tb, wf, wd);
    } else if (fast == 1 || !hs.redo) {
      r = ssa_window<KIND, FilterWide<KIND>>(u, kf, node, Td, tag, k0, k1, tb, wf, wd);
    }
  }
  if (r == SSA_DONE) {
    __syncwarp();
    if (lane == 0) {
#pragma unroll
      for (int p = 0; p < C; ++p) hs.u[p] = u[p];
      hs.code = 0;
      fired += wf;
      drawn += wd;
    }
    __syncwarp();
    return;
  }
  if (KIND == SG_GENERIC || fast) {
    bool done = false;
    while (!done && code == 0) {
      const U4 x = philox10(U4{c + (uint32_t)lane, node, Td, tag}, k0, k1);
      const double nE = -log_pos(u01_open(x.x, x.y));
      // walk the transitions; stop early once the day is surely over
      const float e_lo = itv_neglog(x.x, x.y).lo;
      const float left = (float)(Tn - t) * (1.0f + 0x1.0p-20f);
      int us[C], end[C], walked;
#pragma unroll
      for (int p = 0; p < C; ++p) us[p] = u[p];
      bool open;
      Filter<KIND> N;
      if (fast == 1 && N.load(u, kf, tb)) {
        // 32 transitions leave the counts below 2^24
        open = walk_draws<KIND>(N, x, e_lo, left, kf, tb, us, walked);
#pragma unroll
        for (int p = 0; p < C; ++p) end[p] = (int)N.x[p];
      } else {
        FilterWide<KIND> W;
        W.load(u, kf, tb);
        open = walk_draws<KIND>(W, x, e_lo, left, kf, tb, us, walked);
#pragma unroll
        for (int p = 0; p < C; ++p) end[p] = W.x[p];
      }
      // lane l < walked: draw c + l exactly
      double w[T];
      bool bad = false;
#pragma unroll
      for (int j = 0; j < T; ++j) {
        w[j] = M::rate_k(j, us, kf, tb.gdata);
        bad = bad || bad_rate(w[j]);
      }
      double lam = w[0];
#pragma unroll
      for (int j = 1; j < T; ++j) lam = lam + w[j];
      const double tau = nE / (gt0(lam) ? lam : 1.0);  // unused where lambda = 0
      const unsigned pos_mask = __ballot_sync(full, gt0(lam));
      const unsigned bad_mask = __ballot_sync(full, bad);
      int l = 0;
      for (; l < walked; ++l) {
        if ((bad_mask >> l) & 1u) {
          code = SG_ERR_RATE;  // the transition into this state gave a bad rate
          break;
        }
        if (!((pos_mask >> l) & 1u)) {
          done = true;  // nothing can fire: jump to Tn
          break;
        }
        if (c >= SG_MAX_DRAWS) {
          code = SG_ERR_STEP_LIMIT;
          break;
        }
        const double tt = t + __shfl_sync(full, tau, l);
        ++c;
        if (order_key(tt) >= Tkey) {
          done = true;
          break;
        }
        t = tt;
        ++f;
      }
      if (l < walked || !open) {
        // the counts before draw l (the last walked one if the walk ended
        // there although its event still falls into the day)
        const int src = l < walked ? l : walked - 1;
#pragma unroll
        for (int p = 0; p < C; ++p) u[p] = __shfl_sync(full, us[p], src);
        if (l == walked) {
          // the event of the last draw, which the walk left out
          const uint32_t w2 = __shfl_sync(full, x.z, src), w3 = __shfl_sync(full, x.w, src);
          const int n = select_exact<KIND>(u, kf, w2, w3, tb);
#pragma unroll
          for (int p = 0; p < C; ++p) u[p] += tb.S[n][p];
        }
      } else {
#pragma unroll
        for (int p = 0; p < C; ++p) u[p] = end[p];
      }
    }
  } else {
    double w[T];
#pragma unroll
    for (int j = 0; j < T; ++j) {
      w[j] = M::rate_k(j, u, kf, tb.gdata);
      if (bad_rate(w[j])) code = SG_ERR_RATE;
    }
    uint32_t c0 = c;
    double nE = 0.0, r2 = 0.0;
    bool have = false;
    while (code == 0) {
      double lam = w[0];
#pragma unroll
      for (int j = 1; j < T; ++j) lam = lam + w[j];
      if (!gt0(lam)) break;
      if (c >= SG_MAX_DRAWS) {
        code = SG_ERR_STEP_LIMIT;
        break;
      }
      if (!have || c - c0 >= 32u) {
        c0 = c;
        const U4 x = philox10(U4{c0 + (uint32_t)lane, node, Td, tag}, k0, k1);
        nE = -log_pos(u01_open(x.x, x.y));
        r2 = u01_open(x.z, x.w);
        have = true;
      }
      const int jj = (int)(c - c0);
      const double E = __shfl_sync(full, nE, jj);
      const double R2 = __shfl_sync(full, r2, jj);
      ++c;
      const double tt = t + E / lam;
      if (order_key(tt) >= Tkey) break;
      t = tt;
      code = fire<KIND>(u, w, lam * R2, kf, tb);
      ++f;
    }
  }
  __syncwarp();
  if (lane == 0) {
#pragma unroll
    for (int p = 0; p < C; ++p) hs.u[p] = u[p];
    hs.code = code;
    fired += f;
    drawn += c;
  }
  __syncwarp();
}

// ---------------------------------------------------------------------------
// The all events method (solver 'aem' of Sec. 3.4.2): every transition of a
// node is a channel with its own random stream, Philox counter (draws taken
// by the channel, node, transition, (3 << 24) | replicate), and the channels
// advance by the next reaction method of Gibson and Bruck: each holds an
// absolute firing time, the earliest fires, the fired channel draws a fresh
// Exp(1) waiting time scaled by its rate, a channel whose rate changes from
// a > 0 to a' > 0 rescales its residual time by a / a', one whose rate drops
// to 0 sleeps (time +inf), one that wakes draws afresh.  Firing times carry
// over from day to day; at each day start every rate is recomputed and the
// same rule applied.
// ---------------------------------------------------------------------------

__device__ __forceinline__ int aem_draw(uint32_t &c, uint32_t node, uint32_t j, uint32_t tag,
                                        uint32_t k0, uint32_t k1, double &E) {
  if (c == 0xffffffffu) return SG_ERR_STEP_LIMIT;
  const U4 x = philox10(U4{c, node, j, tag}, k0, k1);
  ++c;
  E = -log_pos(u01_open(x.x, x.y));
  return 0;
}

// a == b for rates (no NaN), by integer instructions: an FP64 comparison
// holds the FP64 pipe as long as any FP64 operation.
__device__ __forceinline__ bool same_rate(double a, double b) {
  const unsigned long long x = (unsigned long long)__double_as_longlong(a);
  const unsigned long long y = (unsigned long long)__double_as_longlong(b);
  return x == y || ((x | y) << 1) == 0ull;
}

// Channel j's new rate a_new at time t (the update rule above).
__device__ __forceinline__ int aem_update(double t, double a_new, double &a, double &tau,
                                          uint32_t &c, uint32_t node, uint32_t j, uint32_t tag,
                                          uint32_t k0, uint32_t k1, unsigned long long &drawn) {
  if (same_rate(a_new, a)) return 0;
  if (gt0(a) && gt0(a_new)) {
    tau = t + (a / a_new) * (tau - t);
  } else if (gt0(a_new)) {
    double E;
    const int rc = aem_draw(c, node, j, tag, k0, k1, E);
    if (rc) return rc;
    ++drawn;
    tau = t + E / a_new;
  } else {
    tau = __longlong_as_double(0x7ff0000000000000ll);  // +inf
  }
  a = a_new;
  return 0;
}

// Day start (t = Tn - 1): every rate recomputed, the update rule applied.
template <int KIND>
__device__ __forceinline__ int aem_day_start(const int *u, const double *kf, double *a,
                                             double *tau, uint32_t *c, double Tn, uint32_t node,
                                             uint32_t tag, uint32_t k0, uint32_t k1,
                                             const SgTables &tb, unsigned long long &drawn) {
  using M = ModelTraits<KIND>;
  const double t = Tn - 1.0;
#pragma unroll
  for (int j = 0; j < M::T; ++j) {
    const double w = M::rate_k(j, u, kf, tb.gdata);
    if (bad_rate(w)) return SG_ERR_RATE;
    const int rc = aem_update(t, w, a[j], tau[j], c[j], node, (uint32_t)j, tag, k0, k1, drawn);
    if (rc) return rc;
  }
  return 0;
}

enum { AEM_DONE = 0, AEM_HEAVY = 1 };

// The earliest channel (ties to the lowest index); -1 if all sleep.
template <int T>
__device__ __forceinline__ int aem_earliest(const double *tau, double &best) {
  int mu = -1;
  best = __longlong_as_double(0x7ff0000000000000ll);
#pragma unroll
  for (int j = 0; j < T; ++j) {
    if (order_key(tau[j]) < order_key(best)) {
      best = tau[j];
      mu = j;
    }
  }
  return mu;
}

// Firings of one node until Tn, at most `budget` of them in this call.  The
// fired channel and the woken ones take their Exp(1) draws from `draw(j,
// E)` (computed on the spot by a thread, from a lane table by a warp).
// Returns AEM_DONE, AEM_HEAVY (budget spent; state ready for a warp) or an
// error.
template <int KIND, typename Draw>
__device__ __forceinline__ int aem_steps(int *u, const double *kf, double *a, double *tau,
                                         uint32_t *c, double &t, uint32_t &nfired, double Tn,
                                         const SgTables &tb, unsigned long long &fired,
                                         int budget, Draw &&draw) {
  using M = ModelTraits<KIND>;
  constexpr int T = M::T;
  const double inf = __longlong_as_double(0x7ff0000000000000ll);
  for (int b = 0;; ++b) {
    double best;
    const int mu = aem_earliest<T>(tau, best);
    if (mu < 0 || order_key(best) >= order_key(Tn)) return AEM_DONE;
    if (nfired >= SG_MAX_DRAWS) return SG_ERR_STEP_LIMIT;
    if (b == budget) return AEM_HEAVY;
    ++nfired;
    t = best;
#pragma unroll
    for (int p = 0; p < M::C; ++p) u[p] += tb.S[mu][p];
    ++fired;
    const uint32_t dep = tb.dep[mu];
#pragma unroll
    for (int k = 0; k < T; ++k) {
      const bool marked = (dep >> k) & 1u;
      if (k != mu && !marked) continue;
      double w = a[k];
      if (marked) {
        w = M::rate_k(k, u, kf, tb.gdata);
        if (bad_rate(w)) return SG_ERR_RATE;
      }
      if (k == mu) {
        // the fired channel always redraws
        a[k] = w;
        if (gt0(w)) {
          double E;
          const int rc = draw(k, E);
          if (rc) return rc;
          tau[k] = t + E / w;
        } else {
          tau[k] = inf;
        }
      } else if (!same_rate(w, a[k])) {
        if (gt0(a[k]) && gt0(w)) {
          tau[k] = t + (a[k] / w) * (tau[k] - t);
        } else if (gt0(w)) {
          double E;
          const int rc = draw(k, E);
          if (rc) return rc;
          tau[k] = t + E / w;
        } else {
          tau[k] = inf;
        }
        a[k] = w;
      }
    }
  }
}

// A node handed from its thread to a warp (all events method).
template <int C, int NK, int T>
struct AemSlot {
  double kf[NK];
  double a[T], tau[T];
  uint32_t c[T];
  uint32_t nfired;
  int32_t node, rep, code;
  int32_t u[C];
};

// Shared-memory slots for hand-offs (at most 24 KB, at most one per thread).
template <int C, int NK, int T>
struct AemSlots {
  static constexpr int n = (int)(24576 / sizeof(AemSlot<C, NK, T>)) < kDayBlock
                               ? (int)(24576 / sizeof(AemSlot<C, NK, T>))
                               : kDayBlock;
};

// The rest of a node-day by a whole warp.  Every channel's next draws depend
// only on its counter, so lane l holds the Exp(1) value of draw c_j +
// (l mod B) of channel j = l / B (B = 32 / T lanes per channel), all computed
// at once; when a channel has used its B values the table is recomputed from
// the current counters.  Lane j < T also holds channel j's rate, firing time
// and counter: after a firing the channels that change (the fired one with
// its new draw, the others by the rescaling rule) share one FP64 division and
// three more operations, and the earliest channel is found by integer
// comparison.  Bound by the FP64 pipe, 14 operations a firing of two channels
// (one channel after the other 30): 1,600 SISe herds x 365 days 13.9 ms, by one
// channel after the other 18.4 ms.  Same operations on every value, in the
// same order, as the thread path.
template <int KIND>
__device__ void aem_warp(AemSlot<ModelTraits<KIND>::C, ModelTraits<KIND>::NK,
                                 ModelTraits<KIND>::T> &hs,
                         double Tn, uint32_t k0, uint32_t k1, const SgTables &tb,
                         unsigned long long &fired, unsigned long long &drawn) {
  using M = ModelTraits<KIND>;
  constexpr int C = M::C, T = M::T, NK = M::NK;
  constexpr int B = 32 / T;
  constexpr unsigned full = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  const int jl = lane / B, il = lane - jl * B;
  const bool mine = lane < T;  // this lane holds channel `lane`
  int u[C];
  double kf[NK];
#pragma unroll
  for (int p = 0; p < C; ++p) u[p] = hs.u[p];
#pragma unroll
  for (int i = 0; i < NK; ++i) kf[i] = hs.kf[i];
  double a = mine ? hs.a[lane] : 0.0;
  double tau = mine ? hs.tau[lane] : 0.0;
  uint32_t c = mine ? hs.c[lane] : 0u;
  int used = B;  // no table yet
  uint32_t nfired = hs.nfired;
  const uint32_t node = (uint32_t)hs.node;
  const uint32_t tag = (SG_STREAM_AEM << 24) | (uint32_t)hs.rep;
  const long long Tkey = order_key(Tn), never = 0x7ff0000000000000ll;
  double myE = 0.0;
  unsigned long long f = 0, dr = 0;
  int code = 0;
  for (;;) {
    const long long key = order_key(tau);
    long long best = never;
    int mu = -1;
#pragma unroll
    for (int j = 0; j < T; ++j) {
      const long long k = __shfl_sync(full, key, j);
      if (k < best) {
        best = k;
        mu = j;
      }
    }
    if (mu < 0 || best >= Tkey) break;
    if (nfired >= SG_MAX_DRAWS) {
      code = SG_ERR_STEP_LIMIT;
      break;
    }
    ++nfired;
    const double t = __shfl_sync(full, tau, mu);
#pragma unroll
    for (int p = 0; p < C; ++p) u[p] += tb.S[mu][p];
    ++f;
    const uint32_t dep = tb.dep[mu];
    double w = a;
    bool bad = false;
#pragma unroll
    for (int k = 0; k < T; ++k) {
      if ((dep >> k) & 1u) {
        const double x = M::rate_k(k, u, kf, tb.gdata);
        bad = bad || bad_rate(x);
        if (lane == k) w = x;
      }
    }
    if (bad) {
      code = SG_ERR_RATE;
      break;
    }
    const bool changes = mine && (lane == mu || !same_rate(w, a));
    const bool awake = changes && gt0(w);
    // the fired channel and the ones that wake take a draw
    const bool draws = awake && (lane == mu || !gt0(a));
    if (__any_sync(full, draws && c == 0xffffffffu)) {
      code = SG_ERR_STEP_LIMIT;
      break;
    }
    if (__any_sync(full, draws && used == B)) {
      const uint32_t cl = __shfl_sync(full, c, jl < T ? jl : 0);
      const uint32_t ci = cl + (uint32_t)il;
      // draws past the counter's end are never used (the check above stops
      // first); compute something harmless for them
      const U4 x = philox10(U4{ci < cl ? cl : ci, node, (uint32_t)jl, tag}, k0, k1);
      myE = -log_pos(u01_open(x.x, x.y));
      used = 0;
    }
    const double E = __shfl_sync(full, myE, (lane * B + used) & 31);
    if (draws) {
      ++c;
      ++used;
    }
    dr += __popc(__ballot_sync(full, draws));
    // lanes without a change divide 1 by 1: an operand of zero in any lane
    // sends the warp through the division's slow path
    const double q = (draws ? E : awake ? a : 1.0) / (awake ? w : 1.0);
    const double step = draws ? q : q * (tau - t);
    const double next = t + step;
    if (changes) {
      tau = awake ? next : __longlong_as_double(never);
      a = w;
    }
  }
  if (mine) {
    hs.a[lane] = a;
    hs.tau[lane] = tau;
    hs.c[lane] = c;
  }
  if (lane == 0) {
#pragma unroll
    for (int p = 0; p < C; ++p) hs.u[p] = u[p];
    hs.code = code;
    fired += f;
    drawn += dr;
  }
  __syncwarp();
}

// The fields of one planned event and the first Philox block of its word
// stream (a function of the seed, the list index and the replicate only), so
// that they can be fetched and computed ahead of the event.
struct E1Rec {
  int type, n, shift, next;
  uint32_t mask;
  long long idx;
  double prop;
  U4 first;
};

__device__ __forceinline__ E1Rec load_e1(const SgTables &tb, const EvDev &ev, long long j, int rep,
                                         uint32_t k0, uint32_t k1) {
  E1Rec r;
  const SgEvent e = load_event(ev.rec + j);
  r.type = e.type;
  r.mask = tb.Emask[e.select];
  r.n = e.n;
  r.shift = e.shift;
  r.next = e.next;
  r.idx = e.index;
  r.prop = e.proportion;
  r.first = philox10(U4{0u, (uint32_t)(unsigned long long)r.idx,
                        (uint32_t)((unsigned long long)r.idx >> 32),
                        (SG_STREAM_EVENTS << 24) | (uint32_t)rep},
                     k0, k1);
  return r;
}

// One E1 event (exit, enter or internal transfer, Sec. 3.3) on a node whose
// counts are in the calling thread's registers.  Returns 0 or an error.
template <int C>
__device__ __forceinline__ int apply_e1(int *u, const SgTables &tb, const E1Rec &e, int rep,
                                        uint32_t k0, uint32_t k1) {
  const int type = e.type;
  const uint32_t mask = e.mask;
  const int n = e.n;
  if (type == SG_ENTER) {
    const int first = __ffs(mask) - 1;  // first selected compartment
#pragma unroll
    for (int p = 0; p < C; ++p)
      if (p == first) u[p] += n;
    return 0;
  }
  long long total = 0;
#pragma unroll
  for (int p = 0; p < C; ++p)
    if ((mask >> p) & 1u) total += u[p];
  const long long k = n > 0 ? (long long)n : (long long)round(e.prop * (double)total);
  if (k < 0 || k > total) return SG_ERR_EVENT_UNDERFLOW;
  int moved[C];
#pragma unroll
  for (int p = 0; p < C; ++p) moved[p] = 0;
  if (k > 0) {
    WordStream ws;
    ws.init_with_first(((uint64_t)k1 << 32) | k0, e.idx, rep, e.first);
    for (long long i = 0; i < k; ++i) {
      uint32_t x = ws.below((uint32_t)(total - i));
      bool taken = false;
#pragma unroll
      for (int p = 0; p < C; ++p) {
        if (taken || !((mask >> p) & 1u)) continue;
        const uint32_t rem = (uint32_t)(u[p] - moved[p]);
        if (x < rem) {
          ++moved[p];
          taken = true;
        } else {
          x -= rem;
        }
      }
    }
  }
#pragma unroll
  for (int p = 0; p < C; ++p) u[p] -= moved[p];
  if (type == SG_EXIT) return 0;
  const int q = e.shift;  // internal transfer: validated q >= 0
#pragma unroll
  for (int dst = 0; dst < C; ++dst) {
    int add = 0;
#pragma unroll
    for (int p = 0; p < C; ++p)
      if (p + tb.Nsh[q][p] == dst) add += moved[p];
    u[dst] += add;
  }
  return 0;
}

// The number of individuals an E1 event draws (exit or internal transfer;
// 0 for an enter, -1 for one that moves more than exist).
template <int C>
__device__ __forceinline__ long long e1_draws(const int *u, const SgTables &tb, const E1Rec &e) {
  if (e.type == SG_ENTER) return 0;
  long long total = 0;
#pragma unroll
  for (int p = 0; p < C; ++p)
    if ((e.mask >> p) & 1u) total += u[p];
  const long long k = e.n > 0 ? (long long)e.n : (long long)round(e.prop * (double)total);
  return (k < 0 || k > total) ? -1 : k;
}

// The E1 event `e` of lane `owner` (an exit or internal transfer drawing at
// least kUrnWarp individuals), applied by the whole warp: the owner's counts
// and event fields are broadcast, the warp samples the urn (urn_warp, the
// same draws as apply_e1), and the owner's counts are updated.  Every lane
// calls it with the same owner; returns the owner's result in every lane.
template <int C>
__device__ __forceinline__ int apply_e1_warp(int *u, const SgTables &tb, const E1Rec &e,
                                             int owner, int rep, uint32_t k0, uint32_t k1) {
  const int lane = threadIdx.x & 31;
  int cu[C];
#pragma unroll
  for (int p = 0; p < C; ++p) cu[p] = __shfl_sync(0xffffffffu, u[p], owner);
  const int type = __shfl_sync(0xffffffffu, e.type, owner);
  const uint32_t mask = __shfl_sync(0xffffffffu, e.mask, owner);
  const int n = __shfl_sync(0xffffffffu, e.n, owner);
  const int shift = __shfl_sync(0xffffffffu, e.shift, owner);
  const long long idx = __shfl_sync(0xffffffffu, e.idx, owner);
  const double prop = __shfl_sync(0xffffffffu, e.prop, owner);
  const int r = __shfl_sync(0xffffffffu, rep, owner);
  long long total = 0;
#pragma unroll
  for (int p = 0; p < C; ++p)
    if ((mask >> p) & 1u) total += cu[p];
  const long long k = n > 0 ? (long long)n : (long long)round(prop * (double)total);
  if (k < 0 || k > total) return SG_ERR_EVENT_UNDERFLOW;
  int moved[C];
  urn_warp<C>(cu, mask, (uint32_t)k, (uint32_t)total, ((uint64_t)k1 << 32) | k0, idx, r, moved);
  if (lane == owner) {
#pragma unroll
    for (int p = 0; p < C; ++p) u[p] -= moved[p];
    if (type != SG_EXIT) {
#pragma unroll
      for (int dst = 0; dst < C; ++dst) {
        int add = 0;
#pragma unroll
        for (int p = 0; p < C; ++p)
          if (p + tb.Nsh[shift][p] == dst) add += moved[p];
        u[dst] += add;
      }
    }
  }
  return 0;
}

// The E1 events of day index d of the unit of every lane with `pend`, in
// (time, type, list index) order, from its next one `e` on (already loaded).
// Warp-uniform: all 32 lanes call it.  Every round each lane with an event
// left takes it, applied in the thread or (kUrnWarp or more individuals
// drawn) by the whole warp.  ecur and next_day move along the node's list.
// Returns the lane's error code (0 if none; e is then the event).
template <int C>
__device__ __forceinline__ int e1_events(bool pend, E1Rec &e, int *u, long long &ecur,
                                         int &next_day, int d, const SgTables &tb,
                                         const EvDev &ev, int rep, uint32_t k0, uint32_t k1,
                                         unsigned long long &applied) {
  const int lane = threadIdx.x & 31;
  int code = 0;
  while (__any_sync(0xffffffffu, pend)) {
    const bool heavy = pend && e1_draws<C>(u, tb, e) >= kUrnWarp;
    if (pend && !heavy) code = apply_e1<C>(u, tb, e, rep, k0, k1);
    unsigned hm = __ballot_sync(0xffffffffu, heavy);
    while (hm) {
      const int L = __ffs(hm) - 1;
      hm &= hm - 1;
      const int rc = apply_e1_warp<C>(u, tb, e, L, rep, k0, k1);
      if (lane == L) code = rc;
    }
    if (pend) {
      if (code == 0) {
        ++applied;
        ++ecur;
        next_day = e.next;
      }
      pend = code == 0 && next_day == d;
      if (pend) e = load_e1(tb, ev, ecur, rep, k0, k1);
    }
  }
  return code;
}

// Post time step and recording for unit time Tf (the state after its
// events).  Returns 0 or SG_ERR_PTS.
template <int KIND>
__device__ __forceinline__ int finish_step(int Tf, const int *u, double *v, const int *ends,
                                           const SgTables &tb, const DayArgs &a, int rep,
                                           int node) {
  using M = ModelTraits<KIND>;
  int code = 0;
  if (M::NV > 0) {
    const int r = post_step<KIND>(v, u, ends, tb.gdata, Tf);
    if (r < 0) code = r;
  }
  const int m = a.rec[Tf - a.t0];
  if (m >= 0) {
    const long long base = ((long long)rep * a.M + m) * tb.n_nodes + node;
    if (a.U) {
#pragma unroll
      for (int p = 0; p < M::C; ++p) a.U[base * M::C + p] = u[p];
    }
    if (a.V) {
#pragma unroll
      for (int q = 0; q < M::NV; ++q) a.V[base * M::NV + q] = v[q];
    }
    record_sparse<M::C, M::NV>(a.out, m, rep, node, u, v);
  }
  return code;
}

// The day kernel: one thread per (replicate, node) for a run of days
// T_begin .. T_end - 1 with no external transfers before T_end - 1.  Per day:
// rates, SSA (thread, then warp for heavy nodes), the node's E1 events, and
// (unless a kernel boundary follows) the post time step and recording.
template <int KIND, bool AEM>
__global__ void __launch_bounds__(kDayBlock)
k_days(const __grid_constant__ SgTables tb, const __grid_constant__ DayArgs a) {
  using M = ModelTraits<KIND>;
  constexpr int C = M::C, T = M::T, NV = M::NV, NK = M::NK;
  __shared__ HeavySlot<C, NK> s_heavy[AEM ? 1 : kDayBlock];
  constexpr int kAemSlots = AEM ? AemSlots<C, NK, T>::n : 1;
  __shared__ AemSlot<C, NK, T> s_aheavy[kAemSlots];
  __shared__ int s_nheavy;
  pdl_trigger();
  const int Nn = tb.n_nodes;
  const long long gid = (long long)blockIdx.x * a.npb + threadIdx.x;
  const long long total = (long long)Nn * a.n_rep;
  const bool in_range = (int)threadIdx.x < a.npb && gid < total;
  const int warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
  unsigned long long fired = 0, drawn = 0, applied = 0;
  int rep = 0, node = 0, code = 0, bad_day = 0;
  long long bad_event = -1;
  int u[C];
  double v[NV > 0 ? NV : 1];
  int ld[4] = {0, 0, 0, 0};  // season ends of the node (integer form)
#pragma unroll
  for (int p = 0; p < C; ++p) u[p] = 0;
  v[0] = 0.0;
  long long ecur = 0, ebase = 0;
  int next_day = SG_NO_DAY;
  double ch_a[AEM ? T : 1], ch_tau[AEM ? T : 1];  // all events method channels
  uint32_t ch_c[AEM ? T : 1];
  // static inputs first (they overlap the previous kernel's tail)
  if (in_range) {
    rep = (int)(gid / Nn);
    node = (int)(gid - (long long)rep * Nn);
    if (NV > 0) load_ends(a.ends, a.ldata, tb, node, ld);
    if (a.ev.e1_node_off) {
      const long long key = (long long)(a.slots > 1 ? rep : 0) * Nn + node;
      ebase = a.ev.e1_node_off[key];
    }
  }
  pdl_wait();
  bool live = in_range && *(volatile int32_t *)&a.err->code == 0;
  if (live && a.emu_part == 1) live = a.emu_flag[gid] == 0;
  if (live && a.emu_part == 2) live = a.emu[gid * 4 + 3] != 0;
  if (live) {
#pragma unroll
    for (int p = 0; p < C; ++p) u[p] = a.u[gid * C + p];
#pragma unroll
    for (int q = 0; q < NV; ++q) v[q] = a.v[gid * NV + q];
    if (a.ev.e1_node_off) {
      ecur = ebase + a.e1_cur[gid];
      next_day = a.e1_next[gid];
    }
    if constexpr (AEM) {
#pragma unroll
      for (int j = 0; j < T; ++j) {
        ch_a[j] = a.aem_a[j * total + gid];
        ch_tau[j] = a.aem_tau[j * total + gid];
        ch_c[j] = a.aem_cnt[j * total + gid];
      }
    }
    if (a.finish_first) {
      code = finish_step<KIND>(a.T_begin - 1, u, v, ld, tb, a, rep, node);
      if (code) bad_day = a.T_begin - 1;
    }
  }
  if (a.finish_first && a.out.prev) {
    const int m = a.rec[a.T_begin - 1 - a.t0];
    if (m >= 0)
      prevalence_add<C>(a.out, in_range ? (long long)rep * a.M + m : -1, live && code == 0, u);
  }
  const int grep = a.rep0 + rep;  // global replicate: streams, error reports
  const uint32_t tag = (SG_STREAM_SSA << 24) | (uint32_t)grep;
  for (int Td = a.T_begin; Td < a.T_end; ++Td) {
    const double Tn = (double)Td;
    if (threadIdx.x == 0) s_nheavy = 0;
    __syncthreads();
    int my = -1;
    // the node's first E1 event of the day: fields and first random block
    // fetched now, so that their latency overlaps the SSA
    const int d = Td - a.t0 - 1;
    const bool e1_today = live && code == 0 && next_day == d;
    E1Rec pre;
    if (e1_today) pre = load_e1(tb, a.ev, ecur, grep, a.k0, a.k1);
    const bool emulated =
        !AEM && live && code == 0 && a.emu != nullptr && a.emu[gid * 4 + 3] != 0;
    if (emulated) {
      // the learned emulator's sampled one-day increments (SISe3 only):
      // I_a += d_a, S_a -= d_a, each age class keeps its size
#pragma unroll
      for (int h = 0; h < C / 2; ++h) {
        const int dlt = a.emu[gid * 4 + h];
        u[2 * h] -= dlt;
        u[2 * h + 1] += dlt;
      }
    }
    if (AEM && live && code == 0) {
      double kf[NK];
      M::prepare(v, tb.gdata, kf);
      const uint32_t tag = (SG_STREAM_AEM << 24) | (uint32_t)grep;
      code = aem_day_start<KIND>(u, kf, ch_a, ch_tau, ch_c, Tn, (uint32_t)node, tag, a.k0, a.k1,
                                 tb, drawn);
      double t = Tn - 1.0;
      uint32_t nfired = 0;
      if (code == 0) {
        auto draw = [&](int j, double &E) -> int {
          uint32_t cj = 0;
#pragma unroll
          for (int q = 0; q < T; ++q)
            if (q == j) cj = ch_c[q];
          const int rc = aem_draw(cj, (uint32_t)node, (uint32_t)j, tag, a.k0, a.k1, E);
#pragma unroll
          for (int q = 0; q < T; ++q)
            if (q == j) ch_c[q] = cj;
          if (rc == 0) ++drawn;
          return rc;
        };
        const int r = aem_steps<KIND>(u, kf, ch_a, ch_tau, ch_c, t, nfired, Tn, tb, fired,
                                      a.heavy_after, draw);
        if (r == AEM_HEAVY) {
          const int slot = atomicAdd(&s_nheavy, 1);
          if (slot < kAemSlots) {
            my = slot;
            AemSlot<C, NK, T> &hs = s_aheavy[slot];
#pragma unroll
            for (int i = 0; i < NK; ++i) hs.kf[i] = kf[i];
#pragma unroll
            for (int j = 0; j < T; ++j) {
              hs.a[j] = ch_a[j];
              hs.tau[j] = ch_tau[j];
              hs.c[j] = ch_c[j];
            }
            hs.nfired = nfired;
            hs.node = node;
            hs.rep = grep;
            hs.code = 0;
#pragma unroll
            for (int p = 0; p < C; ++p) hs.u[p] = u[p];
          } else {
            // no slot left: the thread finishes its node itself
            const int r2 = aem_steps<KIND>(u, kf, ch_a, ch_tau, ch_c, t, nfired, Tn, tb, fired,
                                           -1, draw);
            if (r2 < 0) code = r2;
          }
        } else if (r < 0) {
          code = r;
        }
      }
      if (code) bad_day = Td;
    }
    if constexpr (!AEM) {
      const bool ssa = live && code == 0 && !emulated;
      double kf[NK];
      if (ssa) M::prepare(v, tb.gdata, kf);
      auto to_slot = [&](int redo) {
        HeavySlot<C, NK> &hs = s_heavy[my];
        hs.redo = redo;
#pragma unroll
        for (int i = 0; i < NK; ++i) hs.kf[i] = kf[i];
        hs.node = node;
        hs.rep = grep;
        hs.code = 0;
#pragma unroll
        for (int p = 0; p < C; ++p) hs.u[p] = u[p];
      };
      if (a.fast && ssa) {
        // a long day goes to a warp if the block has few of them
        Itv lambda;
        if (day_rate<KIND>(u, kf, a.fast, tb, lambda) && lambda.lo >= a.warp_rate) {
          my = atomicAdd(&s_nheavy, 1);
          to_slot(0);
        }
      }
      __syncthreads();
      const bool own = s_nheavy > a.warp_max;
      __syncthreads();
      if (ssa && (my < 0 || own)) {
        const int r = ssa_thread<KIND>(u, kf, (uint32_t)node, (uint32_t)Td, tag, a.k0, a.k1,
                                       a.fast, a.heavy_after, tb, fired, drawn);
        if (r == SSA_REDO) {
          if (my < 0) my = atomicAdd(&s_nheavy, 1);
          to_slot(1);
        } else {
          if (my >= 0) s_heavy[my].rep = -1;  // done
          my = -1;
          if (r < 0) code = r;
        }
      }
      if (ssa && code) bad_day = Td;
    }
    __syncthreads();
    if constexpr (!AEM) {
      const int nh = s_nheavy;
      for (int h = warp; h < nh; h += nwarps)
        if (s_heavy[h].rep >= 0)
          ssa_warp<KIND>(s_heavy[h], Tn, (uint32_t)Td, a.k0, a.k1, a.fast, tb, fired, drawn);
    } else {
      const int nh = min(s_nheavy, kAemSlots);
      for (int h = warp; h < nh; h += nwarps)
        aem_warp<KIND>(s_aheavy[h], Tn, a.k0, a.k1, tb, fired, drawn);
    }
    __syncthreads();
    if (AEM && my >= 0) {
#pragma unroll
      for (int p = 0; p < C; ++p) u[p] = s_aheavy[my].u[p];
#pragma unroll
      for (int j = 0; j < T; ++j) {
        ch_a[j] = s_aheavy[my].a[j];
        ch_tau[j] = s_aheavy[my].tau[j];
        ch_c[j] = s_aheavy[my].c[j];
      }
      if (s_aheavy[my].code) {
        code = s_aheavy[my].code;
        bad_day = Td;
      }
      my = -1;
    }
    if (my >= 0) {
#pragma unroll
      for (int p = 0; p < C; ++p) u[p] = s_heavy[my].u[p];
      if (s_heavy[my].code) {
        code = s_heavy[my].code;
        bad_day = Td;
      }
    }
    // this node's E1 events of day Td (every thread of the block gets here)
    {
      const int rc = e1_events<C>(e1_today && code == 0, pre, u, ecur, next_day, d, tb, a.ev,
                                  grep, a.k0, a.k1, applied);
      if (rc) {
        code = rc;
        bad_day = Td;
        bad_event = pre.idx;
      }
    }
    if (a.grid_bar && a.wave_off) {
      // persistent run: the day's external transfers between two grid
      // barriers, by the block holding each replicate's first node, on the
      // state in global memory
      const long long wlo = a.wave_off[(long long)d * a.slots];
      const long long whi = a.wave_off[(long long)(d + 1) * a.slots];
      if (wlo < whi) {  // the same decision in every block
        if (live) {
#pragma unroll
          for (int p = 0; p < C; ++p) a.u[gid * C + p] = u[p];
        }
        __threadfence();
        if (!grid_barrier(a.grid_bar, a.n_blocks, a.err)) break;
        const long long g_lo = (long long)blockIdx.x * a.npb;
        const long long g_hi = min(total, g_lo + a.npb) - 1;
        for (int r = (int)((g_lo + Nn - 1) / Nn); (long long)r * Nn <= g_hi; ++r) {
          // this block holds node 0 of replicate r
          const long long k = (long long)d * a.slots + (a.slots > 1 ? r : 0);
          e2_rep_block<C>(tb, a, r, Td, a.wave_off[k], a.wave_off[k + 1]);
        }
        __threadfence();
        if (!grid_barrier(a.grid_bar, a.n_blocks, a.err)) break;
        if (live) {
#pragma unroll
          for (int p = 0; p < C; ++p) u[p] = __ldcg(a.u + gid * C + p);
        }
      }
    }
    if (live && code == 0 && (Td + 1 < a.T_end || a.finish_last)) {
      code = finish_step<KIND>(Td, u, v, ld, tb, a, rep, node);
      if (code) bad_day = Td;
    }
    if ((Td + 1 < a.T_end || a.finish_last) && a.out.prev) {
      const int m = a.rec[Td - a.t0];
      if (m >= 0)
        prevalence_add<C>(a.out, in_range ? (long long)rep * a.M + m : -1, live && code == 0,
                          u);
    }
  }
  if (live) {
    if (code) report(a.err, code, a.rep0 + rep, node, bad_day, bad_event);
#pragma unroll
    for (int p = 0; p < C; ++p) a.u[gid * C + p] = u[p];
#pragma unroll
    for (int q = 0; q < NV; ++q) a.v[gid * NV + q] = v[q];
    if (a.ev.e1_node_off) {
      a.e1_cur[gid] = (int32_t)(ecur - ebase);
      a.e1_next[gid] = next_day;
    }
    if constexpr (AEM) {
#pragma unroll
      for (int j = 0; j < T; ++j) {
        a.aem_a[j * total + gid] = ch_a[j];
        a.aem_tau[j * total + gid] = ch_tau[j];
        a.aem_cnt[j * total + gid] = ch_c[j];
      }
    }
  }
  if (a.e2_done) {
    // the last block to finish a replicate's nodes runs its external
    // transfers of T_end - 1 (threadfence-reduction pattern: no block waits)
    __shared__ int s_last;
    __threadfence();
    __syncthreads();
    const long long g_lo = (long long)blockIdx.x * a.npb;
    const long long g_hi = min(total, g_lo + a.npb) - 1;
    for (int r = (int)(g_lo / Nn); r <= (int)(g_hi / Nn); ++r) {
      if (threadIdx.x == 0) {
        const long long b_first = (long long)r * Nn / a.npb;
        const long long b_last = ((long long)(r + 1) * Nn - 1) / a.npb;
        const int old = atomicAdd(&a.e2_done[r], 1);
        s_last = old == (int)(b_last - b_first);
      }
      __syncthreads();
      if (s_last) {
        __threadfence();
        long long w0 = a.e2_wb, w1 = a.e2_we;
        if (a.slots > 1) {
          w0 = a.wave_off[(long long)a.e2_day_index * a.slots + r];
          w1 = a.wave_off[(long long)a.e2_day_index * a.slots + r + 1];
        }
        e2_rep_block<C>(tb, a, r, a.T_end - 1, w0, w1);
        if (threadIdx.x == 0) a.e2_done[r] = 0;
      }
      __syncthreads();
    }
  }
  // one atomic per warp for the counters
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    fired += __shfl_down_sync(0xffffffffu, fired, off);
    drawn += __shfl_down_sync(0xffffffffu, drawn, off);
    applied += __shfl_down_sync(0xffffffffu, applied, off);
  }
  if ((threadIdx.x & 31) == 0) {
    if (drawn | fired) {
      atomicAdd(&a.cnt->reactions, fired);
      atomicAdd(&a.cnt->draws, drawn);
    }
    if (applied) atomicAdd(&a.cnt->events, applied);
  }
}

// ---------------------------------------------------------------------------
// Day kernel for sparse activity (the direct method on the built-in kinds).
// On cattle-shaped workloads only a few percent of the node-days have a
// positive total rate; the rest take no draw, and on the thread-per-node
// schedule above their threads still compute every rate and the post time
// step in FP64 (GB300's weakest pipe) and wait at block barriers for the
// block's few active nodes.  Here a block owns a contiguous range of
// `npb` (> kDayBlock) (replicate, node) units whose state stays in global
// memory (L2), and each day it
//   1. visits every unit: finishes the previous day when the launch starts
//      with it, and tests whether the unit's day is certainly empty
//      (quiescent<>: no infected animal and phi exactly +0, with finite
//      parameters every rate is then +-0 and the post time step leaves phi
//      at +0, so skipping them changes no bit); the other units get their
//      rates, and those with lambda > 0 go to a shared list;
//   2. runs the SSA of the listed units, one thread each (dense lanes);
//      days that need exact times go to warps;
//   3. visits every unit again: its E1 events of the day (per-unit cursor)
//      and, unless the day's external transfers follow in their own kernel,
//      the post time step and recording.
// Units are taken in chunks of kSparseChunk so that the list fits in shared
// memory.  Every unit's operations and random draws are the ones of the
// thread-per-node schedule, so the results are identical.
// ---------------------------------------------------------------------------
constexpr int kSparseBlock = 256;   // threads of the sparse-schedule day kernel
constexpr int kSparseChunk = 8192;  // units per pass through the active list
constexpr int kSparseHeavy = 64;    // warp hand-off slots per pass, of which long
constexpr int kSparseDirect = 48;   // days take at most these; the others are for redone days

// A unit whose day is certainly empty: no infected animal and phi == +0
// (bit pattern 0).  Exact only with finite model parameters (DayArgs::quiet).
template <int KIND>
__device__ __forceinline__ bool quiescent(const int *u, const double *v) {
  if constexpr (KIND == SG_SIR || KIND == SG_SIS) {
    return u[1] == 0;
  } else if constexpr (KIND == SG_SISE) {
    return u[1] == 0 && __double_as_longlong(v[0]) == 0;
  } else if constexpr (KIND == SG_SISE3) {
    return (u[1] | u[3] | u[5]) == 0 && __double_as_longlong(v[0]) == 0;
  } else {
    return false;
  }
}

// Recording of a unit whose post time step leaves it unchanged (tspan
// slot m >= 0): dense U / V and the sparse entries.
template <int C, int NV>
__device__ __forceinline__ void record_unit(const DayArgs &a, int Nn, int m, int rep, int node,
                                            const int *u, const double *v) {
  const long long base = ((long long)rep * a.M + m) * Nn + node;
  if (a.U) {
#pragma unroll
    for (int p = 0; p < C; ++p) a.U[base * C + p] = u[p];
  }
  if (a.V) {
#pragma unroll
    for (int q = 0; q < NV; ++q) a.V[base * NV + q] = v[q];
  }
  record_sparse<C, NV>(a.out, m, rep, node, u, v);
}

// Post time step and recording of unit time Tf for one unit of the sparse
// schedule (counts u, continuous state v, stored back); a quiescent unit's
// post time step is skipped (phi stays +0).  Returns 0 or SG_ERR_PTS.
template <int KIND>
__device__ __forceinline__ int sparse_finish(int Tf, const int *u, double *v, bool quiet,
                                             const SgTables &tb, const DayArgs &a, int rep,
                                             int node, long long gid) {
  using M = ModelTraits<KIND>;
  constexpr int C = M::C, NV = M::NV;
  if (quiet && quiescent<KIND>(u, v)) {
    const int m = a.rec[Tf - a.t0];
    if (m >= 0) {
      const long long base = ((long long)rep * a.M + m) * tb.n_nodes + node;
      if (a.U) {
#pragma unroll
        for (int p = 0; p < C; ++p) a.U[base * C + p] = u[p];
      }
      if (a.V) {
#pragma unroll
        for (int q = 0; q < NV; ++q) a.V[base * NV + q] = v[q];
      }
      record_sparse<C, NV>(a.out, m, rep, node, u, v);
    }
    return 0;
  }
  int ld[4] = {0, 0, 0, 0};
  if (NV > 0) load_ends(a.ends, a.ldata, tb, node, ld);
  const int code = finish_step<KIND>(Tf, u, v, ld, tb, a, rep, node);
  if (code) report(a.err, code, a.rep0 + rep, node, Tf, -1);
#pragma unroll
  for (int q = 0; q < NV; ++q) a.v[gid * NV + q] = v[q];
  return code;
}

// E1 events of day index d (unit time Td) of the unit of every lane with
// `has`, whose next event is of that day, for the sparse schedule (state in
// device memory).  Warp-uniform.  Returns the lane's error code (0 if none).
template <int C>
__device__ __forceinline__ int sparse_e1(bool has, long long gid, int rep, int node, int Td,
                                         int d, const SgTables &tb, const DayArgs &a,
                                         uint32_t k0, uint32_t k1,
                                         unsigned long long &applied) {
  const int Nn = tb.n_nodes;
  long long ecur = 0, ebase = 0;
  int u[C], next_day = d;
#pragma unroll
  for (int p = 0; p < C; ++p) u[p] = 0;
  const int grep = a.rep0 + rep;
  E1Rec e;
  if (has) {
    const long long key = (long long)(a.slots > 1 ? rep : 0) * Nn + node;
    ebase = a.ev.e1_node_off[key];
    ecur = ebase + a.e1_cur[gid];
#pragma unroll
    for (int p = 0; p < C; ++p) u[p] = a.u[gid * C + p];
    e = load_e1(tb, a.ev, ecur, grep, k0, k1);
  }
  const int code =
      e1_events<C>(has, e, u, ecur, next_day, d, tb, a.ev, grep, k0, k1, applied);
  if (code) report(a.err, code, grep, node, Td, e.idx);
  if (has) {
#pragma unroll
    for (int p = 0; p < C; ++p) a.u[gid * C + p] = u[p];
    a.e1_cur[gid] = (int32_t)(ecur - ebase);
    a.e1_next[gid] = next_day;
  }
  return code;
}

// E1 events of day Td of the units marked in a chunk's bitmaps: units with
// events today (e1bits) that took SSA draws (actbits) when `act`, else those
// that did not.  A warp takes `words` words (at most 32, of 32 units each) at a time from *take,
// counts the marked units of each word, and gives the k-th marked unit of
// the take to lane k mod 32 in round k / 32 (word by a search over the
// warp's prefix counts, bit by halving), so the lanes stay full however
// sparse the marks are.  Warp-uniform; called by every lane of a warp.
// *failed (shared) is set where an event fails.
template <int C>
__device__ __forceinline__ void sparse_e1_bits(const uint32_t *e1bits, const uint32_t *actbits,
                                               bool act, int *take, int words, int nw,
                                               long long gbase,
                                               int Td, int d, const SgTables &tb,
                                               const DayArgs &a, uint32_t k0, uint32_t k1,
                                               unsigned long long &applied, int *failed) {
  const int lane = threadIdx.x & 31;
  const int Nn = tb.n_nodes;
  for (;;) {
    int g = 0;
    if (lane == 0) g = atomicAdd(take, words);
    g = __shfl_sync(0xffffffffu, g, 0);
    if (g >= nw) break;
    const int wi = g + lane;
    uint32_t m = 0;
    if (lane < words && wi < nw) m = e1bits[wi] & (act ? actbits[wi] : ~actbits[wi]);
    const int cnt = __popc(m);
    int incl = cnt;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, incl, off);
      if (lane >= off) incl += y;
    }
    const int excl = incl - cnt;
    const int tot = __shfl_sync(0xffffffffu, incl, 31);
#pragma unroll 1
    for (int r0 = 0; r0 < tot; r0 += 32) {
      const int k = r0 + lane;
      // the last word whose count starts at or below k
      int w = 0;
#pragma unroll
      for (int sft = 16; sft > 0; sft >>= 1) {
        const int e = __shfl_sync(0xffffffffu, excl, w + sft);
        if (e <= k) w += sft;
      }
      uint32_t x = __shfl_sync(0xffffffffu, m, w);
      int n = k - __shfl_sync(0xffffffffu, excl, w);
      int pos = 0;
#pragma unroll
      for (int sft = 16; sft > 0; sft >>= 1) {
        const int c = __popc(x & ((1u << sft) - 1u));
        if (n >= c) {
          n -= c;
          x >>= sft;
          pos += sft;
        }
      }
      const bool has = k < tot;
      long long gid = 0;
      int rep = 0, node = 0;
      if (has) {
        gid = gbase + (long long)(g + w) * 32 + pos;
        rep = (int)(gid / Nn);
        node = (int)(gid - (long long)rep * Nn);
      }
      if (sparse_e1<C>(has, gid, rep, node, Td, d, tb, a, k0, k1, applied)) *failed = 1;
    }
  }
}

// (replicate, node) of a unit index, advanced by a stride without dividing
// (the passes over a block's units step by kSparseBlock).
struct UnitPos {
  int rep, node;
  __device__ __forceinline__ void set(long long gid, int Nn) {
    rep = (int)(gid / Nn);
    node = (int)(gid - (long long)rep * Nn);
  }
  __device__ __forceinline__ void advance(int by, int Nn) {
    node += by;
    while (node >= Nn) {
      node -= Nn;
      ++rep;
    }
  }
};

// OWN: a caller's own S (DayArgs::fast is 2).  Two kernels, because a third
// branch in the list's loop costs the kind's own tables their registers (256 x
// 5,000 x 60 days 3.6 ms instead of 3.4).
template <int KIND, bool OWN>
__global__ void __launch_bounds__(kSparseBlock, 2)
k_days_sparse(const __grid_constant__ SgTables tb, const __grid_constant__ DayArgs a) {
  using M = ModelTraits<KIND>;
  constexpr int C = M::C, T = M::T, NV = M::NV, NK = M::NK;
  // lists of units of the current chunk (indices relative to the chunk)
  __shared__ uint16_t s_act[kSparseChunk];
  __shared__ uint16_t s_nq[kSparseChunk];  // units of the chunk that are not quiescent
  __shared__ HeavySlot<C, NK> s_heavy[kSparseHeavy];
  __shared__ uint32_t s_actbits[kSparseChunk / 32];  // units taking SSA draws today
  __shared__ uint32_t s_e1bits[kSparseChunk / 32];   // units with E1 events today
  __shared__ int s_nact, s_nheavy, s_stop, s_next, s_nnq, s_e1take, s_e1late, s_nshort, s_nredo;
  __shared__ int s_failed;  // a unit of the block met an error today
  __shared__ __align__(16) E2Stage s_e2;  // the day's transfers of the block's first replicate
  pdl_trigger();
  const int Nn = tb.n_nodes;
  const long long total = (long long)Nn * a.n_rep;
  const long long g0 = (long long)blockIdx.x * a.npb;
  const int nub = (int)max(0LL, min((long long)a.npb, total - g0));
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarps = blockDim.x >> 5;
  const bool quiet = a.quiet != 0;
  const bool has_e1 = a.ev.e1_node_off != nullptr;
  const uint32_t k0 = a.k0, k1 = a.k1;
  unsigned long long rated = 0;  // units whose rates this thread evaluated
  unsigned long long fired = 0, drawn = 0, applied = 0;
  pdl_wait();
  if (a.finish_first && a.T_begin >= a.T_end &&
      *(volatile int32_t *)&a.err->code == 0) {
    // a launch that only finishes unit time T_begin - 1 (the run's last
    // step after its external transfers)
    const int Tf = a.T_begin - 1;
    UnitPos pos;
    pos.set(g0 + tid, Nn);
    for (int i0 = 0; i0 < nub; i0 += kSparseBlock, pos.advance(kSparseBlock, Nn)) {
      const int i = i0 + tid;
      const bool in = i < nub;
      const long long gid = g0 + i;
      int u[C];
      double v[NV > 0 ? NV : 1];
      int rep = 0, node = 0, code = 0;
      v[0] = 0.0;
#pragma unroll
      for (int p = 0; p < C; ++p) u[p] = 0;
      if (in) {
        rep = pos.rep;
        node = pos.node;
#pragma unroll
        for (int p = 0; p < C; ++p) u[p] = a.u[gid * C + p];
#pragma unroll
        for (int q = 0; q < NV; ++q) v[q] = a.v[gid * NV + q];
        code = sparse_finish<KIND>(Tf, u, v, quiet, tb, a, rep, node, gid);
      }
      if (a.out.prev) {
        const int m = a.rec[Tf - a.t0];
        if (m >= 0)
          prevalence_add<C>(a.out, in ? (long long)rep * a.M + m : -1, in && code == 0, u);
      }
    }
  }
  for (int Td = a.T_begin; Td < a.T_end; ++Td) {
    // a failed run stops at the next day boundary (the block's verdict)
    if (tid == 0) {
      s_stop = *(volatile int32_t *)&a.err->code != 0;
      s_failed = 0;
    }
    __syncthreads();
    if (s_stop) break;
    const double Tn = (double)Td;
    const int d = Td - a.t0 - 1;
    // the post time step and recording of Td - 1 in this day's first
    // passes: at a launch that finishes the previous one's last day, and on
    // every day after the first when the block runs its replicates'
    // external transfers itself
    const bool fin_prev = (Td == a.T_begin && a.finish_first) ||
                          (a.e2_inblock && Td > a.T_begin);
    for (int c0 = 0; c0 < nub; c0 += kSparseChunk) {
      const int cn = min(kSparseChunk, nub - c0);
      if (tid == 0) {
        s_nact = 0;
        s_nheavy = 0;
        s_next = 0;
        s_nnq = 0;
        s_e1take = 0;
        s_e1late = 0;
        s_nshort = 0;
        s_nredo = 0;
      }
      for (int q = tid; q < kSparseChunk / 32; q += kSparseBlock) s_actbits[q] = 0u;
      __syncthreads();
      // 1a. every unit of the chunk, four per thread per step (their loads
      //     issued together): a quiescent unit (no infected animal, phi ==
      //     +0) has an empty day and, at the launch's start, only its record
      //     of Td - 1 to write; the others are listed
      const int m_prev = fin_prev ? a.rec[Td - 1 - a.t0] : -1;
      bool paired = false;
      if constexpr (KIND != SG_SIR) {
        // Compartments come in (S, I) pairs and nothing but dense output is
        // recorded: the counts are read and recorded as they lie in memory,
        // 8 bytes a lane, 256 consecutive bytes a warp instruction (a unit
        // per lane touches each 32-byte sector up to six times: 5,000 units
        // of 24 bytes took 14 us a day).  Every unit's counts are recorded
        // here; the post time step of the listed ones changes phi only.
        paired = !a.out.prev && a.out.u_nnz == 0 && a.out.v_nnz == 0 &&
                 (((uintptr_t)a.U) & 7) == 0;
        if (paired) {
          constexpr int H = C / 2;  // pairs of a unit
          UnitPos pos;              // the warp's first unit of the step
          pos.set(g0 + c0 + warp * 32, Nn);
          const int2 *state = reinterpret_cast<const int2 *>(a.u) + (g0 + c0) * H;
#pragma unroll 1
          for (int b0 = 0; b0 < cn; b0 += 4 * kSparseBlock) {
            int2 w[4][H];
            double v[4];
            int nday[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
              const int ub = b0 + k * kSparseBlock + warp * 32, i = ub + lane;
#pragma unroll
              for (int j = 0; j < H; ++j) {
                const int q = j * 32 + lane;
                w[k][j] = make_int2(0, 0);
                if (q < (cn - ub) * H) w[k][j] = state[(long long)ub * H + q];
              }
              v[k] = 0.0;
              nday[k] = -1;
              if (i < cn) {
                if (NV > 0) v[k] = a.v[g0 + c0 + i];
                if (has_e1) nday[k] = a.e1_next[g0 + c0 + i];
              }
            }
#pragma unroll
            for (int k = 0; k < 4; ++k) {
              const int ub = b0 + k * kSparseBlock + warp * 32, i = ub + lane;
              const bool in = i < cn;
              // one bit per pair with an infected animal; a unit's H bits
              uint32_t inf[3] = {0u, 0u, 0u};
#pragma unroll
              for (int j = 0; j < H; ++j) inf[j] = __ballot_sync(0xffffffffu, w[k][j].y != 0);
              uint32_t mine;
              if (H == 1) {
                mine = (inf[0] >> lane) & 1u;
              } else {
                const int bit = 3 * lane;
                const uint32_t lo = bit < 32 ? inf[0] : bit < 64 ? inf[1] : inf[2];
                const uint32_t hi = bit < 32 ? inf[1] : bit < 64 ? inf[2] : 0u;
                mine = __funnelshift_r(lo, hi, bit & 31) & 7u;
              }
              const bool q0 = in && quiet && mine == 0u && __double_as_longlong(v[k]) == 0;
              const uint32_t bw = __ballot_sync(0xffffffffu, nday[k] == d);
              const uint32_t lw = __ballot_sync(0xffffffffu, in && !q0);
              int at = 0;
              if (lane == 0) {
                if (ub < kSparseChunk) s_e1bits[ub / 32] = bw;
                if (lw) at = atomicAdd(&s_nnq, __popc(lw));
              }
              at = __shfl_sync(0xffffffffu, at, 0);
              if (in && !q0) s_nq[at + __popc(lw & ((1u << lane) - 1u))] = (uint16_t)i;
              if (m_prev >= 0 && ub < cn) {
                // streaming stores: the trajectory leaves the state in L2
                const long long unit =
                    ((long long)pos.rep * a.M + m_prev) * Nn + pos.node;
                if (pos.node + 32 <= Nn) {
                  int2 *U = reinterpret_cast<int2 *>(a.U) + unit * H;
#pragma unroll
                  for (int j = 0; j < H; ++j) {
                    const int q = j * 32 + lane;
                    if (a.U && q < (cn - ub) * H) __stcs(U + q, w[k][j]);
                  }
                  if (NV > 0 && a.V && q0) __stcs(a.V + unit + lane, v[k]);
                } else {
#pragma unroll
                  for (int j = 0; j < H; ++j) {
                    const int q = j * 32 + lane, x = q / H;
                    if (!a.U || ub + x >= cn) continue;
                    UnitPos to = pos;
                    to.advance(x, Nn);
                    reinterpret_cast<int2 *>(
                        a.U)[(((long long)to.rep * a.M + m_prev) * Nn + to.node) * H +
                             (q - x * H)] = w[k][j];
                  }
                  if (NV > 0 && a.V && q0) {
                    UnitPos to = pos;
                    to.advance(lane, Nn);
                    a.V[((long long)to.rep * a.M + m_prev) * Nn + to.node] = v[k];
                  }
                }
              }
              pos.advance(kSparseBlock, Nn);
            }
          }
        }
      }
      if (!paired) {
        UnitPos pos;
        pos.set(g0 + c0 + tid, Nn);
#pragma unroll 1
        for (int b0 = 0; b0 < cn; b0 += 4 * kSparseBlock) {
          int uu[4][C];
          double vv[4][NV > 0 ? NV : 1];
          int nday[4];
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            const int i = b0 + k * kSparseBlock + tid;
            vv[k][0] = 0.0;
            nday[k] = -1;
#pragma unroll
            for (int p = 0; p < C; ++p) uu[k][p] = 0;
            if (i < cn) {
              const long long gid = g0 + c0 + i;
#pragma unroll
              for (int p = 0; p < C; ++p) uu[k][p] = a.u[gid * C + p];
#pragma unroll
              for (int q = 0; q < NV; ++q) vv[k][q] = a.v[gid * NV + q];
              if (has_e1) nday[k] = a.e1_next[gid];
            }
          }
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            const int i = b0 + k * kSparseBlock + tid;
            const bool in = i < cn;
            // a warp's 32 units of step k are one word of the bitmap
            const uint32_t bw = __ballot_sync(0xffffffffu, nday[k] == d);
            if (lane == 0) s_e1bits[(b0 + k * kSparseBlock) / 32 + warp] = bw;
            const bool q0 = in && quiet && quiescent<KIND>(uu[k], vv[k]);
            if (in && !q0) s_nq[atomicAdd(&s_nnq, 1)] = (uint16_t)i;
            if (m_prev >= 0) {
              if (q0) record_unit<C, NV>(a, Nn, m_prev, pos.rep, pos.node, uu[k], vv[k]);
              if (a.out.prev)
                prevalence_add<C>(a.out, in ? (long long)pos.rep * a.M + m_prev : -1, q0,
                                  uu[k]);
            }
            pos.advance(kSparseBlock, Nn);
          }
        }
      }
      __syncthreads();
      // 1b. the listed units: finish of Td - 1 (launch start only), rates;
      //     units with lambda > 0 go to the thread list, or, expecting
      //     warp_rate transitions or more, straight to a warp slot
      {
        const int nq = s_nnq;
#pragma unroll 1
        for (int li = tid; li < nq; li += kSparseBlock) {
          const int i = c0 + s_nq[li];  // block-relative
          const long long gid = g0 + i;
          const int rep = (int)(gid / Nn);
          const int node = (int)(gid - (long long)rep * Nn);
          int u[C];
          double v[NV > 0 ? NV : 1];
          v[0] = 0.0;
#pragma unroll
          for (int p = 0; p < C; ++p) u[p] = a.u[gid * C + p];
#pragma unroll
          for (int q = 0; q < NV; ++q) v[q] = a.v[gid * NV + q];
          int code = 0;
          if (fin_prev) {
            code = sparse_finish<KIND>(Td - 1, u, v, quiet, tb, a, rep, node, gid);
            if (code) s_failed = 1;
            if (a.out.prev && m_prev >= 0 && code == 0)
              prevalence_add_unit<C>(a.out, (long long)rep * a.M + m_prev, u);
          }
          if (code == 0 && !(quiet && quiescent<KIND>(u, v))) {
            ++rated;
            double kf[NK];
            M::prepare(v, tb.gdata, kf);
            // lambda: an interval, or (a caller's own tables) its value
            bool bad = false, fires;
            float lam;
            Filter<KIND> F;
            Itv L[T];
            if (!OWN && a.fast && F.load(u, kf, tb) && F.sums(L, tb) && L[T - 1].hi <= kItvMax) {
              fires = L[T - 1].hi > 0.0f;
              lam = L[T - 1].lo;
            } else {
              double w[T];
#pragma unroll
              for (int j = 0; j < T; ++j) {
                w[j] = M::rate_k(j, u, kf, tb.gdata);
                bad = bad || bad_rate(w[j]);
              }
              double l = w[0];
#pragma unroll
              for (int j = 1; j < T; ++j) l = l + w[j];
              fires = gt0(l);
              lam = (float)l;
            }
            if (bad) {
              report(a.err, SG_ERR_RATE, a.rep0 + rep, node, Td, -1);
              s_failed = 1;
            } else if (fires) {
              atomicOr(&s_actbits[(i - c0) >> 5], 1u << ((i - c0) & 31));
              int slot = kSparseDirect;
              if (!(lam < a.warp_rate)) slot = atomicAdd(&s_nheavy, 1);
              if (slot < kSparseDirect) {
                HeavySlot<C, NK> &hs = s_heavy[slot];
#pragma unroll
                for (int q = 0; q < NK; ++q) hs.kf[q] = kf[q];
                hs.node = node;
                hs.rep = a.rep0 + rep;
                hs.code = i;  // the unit, until the warp reports
                hs.redo = 0;
#pragma unroll
                for (int p = 0; p < C; ++p) hs.u[p] = u[p];
              } else if (lam < 2.0f) {
                // the thread list: units expecting two transitions or more
                // from the front, the others from the back, so that the
                // longer chains start first
                s_act[kSparseChunk - 1 - atomicAdd(&s_nshort, 1)] = (uint16_t)(i - c0);
              } else {
                s_act[atomicAdd(&s_nact, 1)] = (uint16_t)(i - c0);
              }
            }
          }
        }
      }
      __syncthreads();
      const int nw_e1 = (cn + 31) >> 5;
      const int e1_words = min(32, max(2, (nw_e1 + 2 * nwarps - 1) / (2 * nwarps)));
      const int n_long = s_nact;
      const int na = n_long + s_nshort;
      const int n_direct = min(s_nheavy, kSparseDirect);
      if (a.e2_inblock && c0 == 0 && warp == nwarps - 1) {
        const long long k = (long long)d * a.slots + (a.slots > 1 ? g0 / Nn : 0);
        if (nub > 0) e2_stage(s_e2, a, a.wave_off[k], a.wave_off[k + 1]);
      }
      // long days go to warps if there are few of them, else to the list's
      // front
      const bool own = n_direct > a.warp_max;
      const int na_all = own ? na + n_direct : na;
      const int list_warps =
          min((na_all + 31) >> 5, own ? nwarps : nwarps - min(n_direct, nwarps / 2));
      if (warp >= list_warps && !own) {
        for (int h = warp - list_warps; h < n_direct; h += nwarps - list_warps) {
          HeavySlot<C, NK> &hs = s_heavy[h];
          const long long gid = g0 + hs.code;
          __syncwarp();
          ssa_warp<KIND>(hs, Tn, (uint32_t)Td, k0, k1, a.fast, tb, fired, drawn);
          if (lane == 0) {
            if (hs.code) {
              report(a.err, hs.code, hs.rep, hs.node, Td, -1);
              s_failed = 1;
            }
#pragma unroll
            for (int p = 0; p < C; ++p) a.u[gid * C + p] = hs.u[p];
          }
          __syncwarp();
        }
      } else {
        for (;;) {
          int li = atomicAdd(&s_next, 1);
          if (li >= na_all) break;
          int slot = -1;
          if (own) {
            if (li < n_direct) slot = li;
            li -= n_direct;
          }
          const long long gid =
              slot >= 0 ? g0 + s_heavy[slot].code
                        : g0 + c0 + s_act[li < n_long ? li : kSparseChunk - 1 - (li - n_long)];
          const int rep = (int)(gid / Nn);
          const int node = (int)(gid - (long long)rep * Nn);
          const uint32_t tag = (SG_STREAM_SSA << 24) | (uint32_t)(a.rep0 + rep);
          int u[C];
          double v[NV > 0 ? NV : 1], kf[NK];
          v[0] = 0.0;
#pragma unroll
          for (int p = 0; p < C; ++p) u[p] = a.u[gid * C + p];
#pragma unroll
          for (int q = 0; q < NV; ++q) v[q] = a.v[gid * NV + q];
          M::prepare(v, tb.gdata, kf);
          int r;
          if constexpr (OWN)
            r = ssa_filter<KIND, FilterWide<KIND>>(u, kf, (uint32_t)node, (uint32_t)Td, tag, k0,
                                                   k1, tb, fired, drawn);
          else
            r = a.fast ? ssa_filter<KIND>(u, kf, (uint32_t)node, (uint32_t)Td, tag, k0, k1, tb,
                                          fired, drawn)
                       : ssa_exact<KIND>(u, kf, (uint32_t)node, (uint32_t)Td, tag, k0, k1,
                                         a.heavy_after, tb, fired, drawn);
          if (r == SSA_REDO) {
            if (slot < 0) slot = n_direct + atomicAdd(&s_nredo, 1);
            if (slot < kSparseHeavy) {
              HeavySlot<C, NK> &hs = s_heavy[slot];
#pragma unroll
              for (int q = 0; q < NK; ++q) hs.kf[q] = kf[q];
              hs.node = node;
              hs.rep = a.rep0 + rep;
              hs.code = (int32_t)(gid - g0);  // the unit, until the warp reports
              hs.redo = 1;
#pragma unroll
              for (int p = 0; p < C; ++p) hs.u[p] = u[p];
              continue;
            }
            // no slot left: this thread runs the day itself
            r = ssa_exact<KIND>(u, kf, (uint32_t)node, (uint32_t)Td, tag, k0, k1, -1, tb, fired,
                                drawn);
          }
          if (slot >= 0 && slot < kSparseHeavy) s_heavy[slot].rep = -1;  // done
          if (r < 0) {
            report(a.err, r, a.rep0 + rep, node, Td, -1);
            s_failed = 1;
          }
#pragma unroll
          for (int p = 0; p < C; ++p) a.u[gid * C + p] = u[p];
        }
      }
      // a warp with no SSA work left applies the E1 events of day Td of the
      // chunk's units that take no draw today (their units with events
      // compacted onto the lanes; about two takes a warp, so that every warp
      // gets some: a round of events is a chain of memory latencies); the
      // units that take
      // draws come after the SSA (their events follow their day's
      // transitions)
      if (has_e1) sparse_e1_bits<C>(s_e1bits, s_actbits, false, &s_e1take, e1_words, nw_e1,
                                    g0 + c0, Td, d, tb, a, k0, k1, applied, &s_failed);
      __syncthreads();
      // the warp slots not run yet: all of them when every warp had list
      // units, else those the thread list handed over
      const int h0 = list_warps < nwarps && !own ? n_direct : 0;
      const int nh = min(n_direct + s_nredo, kSparseHeavy);
      for (int h = h0 + warp; h < nh; h += nwarps) {
        HeavySlot<C, NK> &hs = s_heavy[h];
        if (hs.rep < 0) continue;
        const long long gid = g0 + hs.code;  // the unit (ssa_warp sets the code)
        __syncwarp();
        ssa_warp<KIND>(hs, Tn, (uint32_t)Td, k0, k1, a.fast, tb, fired, drawn);
        if (lane == 0) {
          if (hs.code) {
            report(a.err, hs.code, hs.rep, hs.node, Td, -1);
            s_failed = 1;
          }
#pragma unroll
          for (int p = 0; p < C; ++p) a.u[gid * C + p] = hs.u[p];
        }
        __syncwarp();
      }
      __syncthreads();
      // 3. E1 events of day Td of the units that took draws today
      if (has_e1) {
        sparse_e1_bits<C>(s_e1bits, s_actbits, true, &s_e1late, e1_words, nw_e1, g0 + c0, Td,
                          d, tb, a, k0, k1, applied, &s_failed);
        __syncthreads();
      }
    }
    if (a.e2_inblock) {
      // this block's replicates' external transfers of Td (the wave plan of
      // day d; no other block touches their nodes); none after an error of
      // one of its units today
      asm volatile("cp.async.wait_all;" ::: "memory");
      __syncthreads();
      bool stop = s_failed != 0;
      for (long long r = g0 / Nn; !stop && nub > 0 && r * Nn < g0 + nub; ++r) {
        long long w0 = s_e2.w0, w1 = s_e2.w1;
        if (a.slots > 1 && r != g0 / Nn) {
          const long long k = (long long)d * a.slots + r;
          w0 = a.wave_off[k];
          w1 = a.wave_off[k + 1];
        }
        if (w0 < w1) stop = e2_rep_block<C>(tb, a, (int)r, Td, w0, w1, &s_e2);
      }
      // a failed transfer ends the run before the day's post time step (of
      // which the next day's check takes care but on the last one)
      if (Td + 1 == a.T_end) {
        if (tid == 0) s_stop = *(volatile int32_t *)&a.err->code != 0;
        __syncthreads();
        if (s_stop) break;
      }
    }
    // then, unless deferred to the next day's first passes or the next
    // launch, the post time step and recording of Td for every unit
    const bool fin = a.e2_inblock ? Td + 1 == a.T_end && a.finish_last
                                  : Td + 1 < a.T_end || a.finish_last;
    if (fin) {
      // post time step and recording of Td: quiescent units are recorded
      // by a scan (four per thread per step), the others listed (chunks of
      // kSparseChunk units) and finished from the list
      const int m_fin = a.rec[Td - a.t0];
      for (int c0 = 0; c0 < nub; c0 += kSparseChunk) {
        const int cn = min(kSparseChunk, nub - c0);
        if (tid == 0) s_nnq = 0;
        __syncthreads();
        UnitPos pos;
        pos.set(g0 + c0 + tid, Nn);
#pragma unroll 1
        for (int b0 = 0; b0 < cn; b0 += 4 * kSparseBlock) {
          int uu[4][C];
          double vv[4][NV > 0 ? NV : 1];
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            const int i = b0 + k * kSparseBlock + tid;
            vv[k][0] = 0.0;
#pragma unroll
            for (int p = 0; p < C; ++p) uu[k][p] = 0;
            if (i < cn) {
              const long long gid = g0 + c0 + i;
#pragma unroll
              for (int p = 0; p < C; ++p) uu[k][p] = a.u[gid * C + p];
#pragma unroll
              for (int q = 0; q < NV; ++q) vv[k][q] = a.v[gid * NV + q];
            }
          }
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            const int i = b0 + k * kSparseBlock + tid;
            const bool in = i < cn;
            const bool q0 = in && quiet && quiescent<KIND>(uu[k], vv[k]);
            if (in && !q0) s_nq[atomicAdd(&s_nnq, 1)] = (uint16_t)i;
            if (m_fin >= 0) {
              if (q0) record_unit<C, NV>(a, Nn, m_fin, pos.rep, pos.node, uu[k], vv[k]);
              if (a.out.prev)
                prevalence_add<C>(a.out, in ? (long long)pos.rep * a.M + m_fin : -1, q0,
                                  uu[k]);
            }
            pos.advance(kSparseBlock, Nn);
          }
        }
        __syncthreads();
        const int nq = s_nnq;
#pragma unroll 1
        for (int li = tid; li < nq; li += kSparseBlock) {
          const long long gid = g0 + c0 + s_nq[li];
          const int rep = (int)(gid / Nn);
          const int node = (int)(gid - (long long)rep * Nn);
          int u[C];
          double v[NV > 0 ? NV : 1];
          v[0] = 0.0;
#pragma unroll
          for (int p = 0; p < C; ++p) u[p] = a.u[gid * C + p];
#pragma unroll
          for (int q = 0; q < NV; ++q) v[q] = a.v[gid * NV + q];
          const int code = sparse_finish<KIND>(Td, u, v, quiet, tb, a, rep, node, gid);
          if (a.out.prev && m_fin >= 0 && code == 0)
            prevalence_add_unit<C>(a.out, (long long)rep * a.M + m_fin, u);
        }
        __syncthreads();
      }
    }
    __syncthreads();
  }
  if (a.e2_done) {
    // the last block to finish a replicate's units runs its external
    // transfers of T_end - 1 (counted per replicate, no block waits)
    __shared__ int s_last;
    __threadfence();
    __syncthreads();
    const long long g_hi = g0 + nub - 1;
    for (int r = (int)(g0 / Nn); nub > 0 && (long long)r * Nn <= g_hi; ++r) {
      if (tid == 0) {
        const long long b_first = (long long)r * Nn / a.npb;
        const long long b_last = ((long long)(r + 1) * Nn - 1) / a.npb;
        const int old = atomicAdd(&a.e2_done[r], 1);
        s_last = old == (int)(b_last - b_first);
      }
      __syncthreads();
      if (s_last) {
        __threadfence();
        long long w0 = a.e2_wb, w1 = a.e2_we;
        if (a.slots > 1) {
          w0 = a.wave_off[(long long)a.e2_day_index * a.slots + r];
          w1 = a.wave_off[(long long)a.e2_day_index * a.slots + r + 1];
        }
        e2_rep_block<C>(tb, a, r, a.T_end - 1, w0, w1);
        if (tid == 0) a.e2_done[r] = 0;
      }
      __syncthreads();
    }
  }
  // one atomic per warp for the counters
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    fired += __shfl_down_sync(0xffffffffu, fired, off);
    drawn += __shfl_down_sync(0xffffffffu, drawn, off);
    applied += __shfl_down_sync(0xffffffffu, applied, off);
    rated += __shfl_down_sync(0xffffffffu, rated, off);
  }
  if ((tid & 31) == 0) {
    if (drawn | fired) {
      atomicAdd(&a.cnt->reactions, fired);
      atomicAdd(&a.cnt->draws, drawn);
    }
    if (applied) atomicAdd(&a.cnt->events, applied);
    if (rated) atomicAdd(&a.cnt->rated, rated);
  }
}

// Day index of each unit's first E1 event (or SG_NO_DAY), the per-unit test
// for "events today" (the E1 cursors start at 0).
__global__ void k_e1_next_init(const int64_t *__restrict__ e1_node_off,
                               const int32_t *__restrict__ e1_day, int Nn, int n_rep,
                               int slots, int32_t *e1_next) {
  const long long total = (long long)Nn * n_rep;
  for (long long g = (long long)blockIdx.x * blockDim.x + threadIdx.x; g < total;
       g += (long long)gridDim.x * blockDim.x) {
    const int rep = (int)(g / Nn), node = (int)(g - (long long)rep * Nn);
    const long long key = (long long)(slots > 1 ? rep : 0) * Nn + node;
    const long long b = e1_node_off[key], e = e1_node_off[key + 1];
    e1_next[g] = b < e ? e1_day[b] : SG_NO_DAY;
  }
}

struct EvArgs {
  EvDev ev;
  int *u;
  int32_t n_rep;
  int32_t rep0;  // global index of local replicate 0 (streams, error reports)
  uint32_t k0, k1;
  int32_t day;  // unit time point T the events run at
  SgDevError *err;
  SgCounters *cnt;
};

// Block-wide copy of n 32-bit words with 16-byte accesses where both ends
// are aligned, several loads in flight per thread.
__device__ __forceinline__ void copy_words(int *dst, const int *src, int n) {
  int head = 0;
  if ((((uintptr_t)dst | (uintptr_t)src) & 15) == 0) {
    const int n4 = n >> 2;
    const int4 *s4 = reinterpret_cast<const int4 *>(src);
    int4 *d4 = reinterpret_cast<int4 *>(dst);
#pragma unroll 4
    for (int i = threadIdx.x; i < n4; i += blockDim.x) d4[i] = s4[i];
    head = n4 << 2;
  }
#pragma unroll 4
  for (int i = head + threadIdx.x; i < n; i += blockDim.x) dst[i] = src[i];
}

constexpr int kE2Cap = 896;      // events staged in shared memory per chunk
constexpr int kE2WaveCap = 128;  // wave bounds staged per chunk

// E2 events of one day: block r runs replicate r's external transfers
// (Sec. 3.3) wave by wave, with a block barrier between waves.  The block
// first stages a chunk of events in shared memory together with the first
// Philox block of each event's random stream (which does not depend on the
// state); with SMEM_STATE the replicate's whole node state is also held in
// shared memory for the day.  Several transfers of one wave may share a
// destination, so additions are atomic; a wave never samples a node that
// another event of the wave touches.
template <int KIND, bool SMEM_STATE>
__global__ void __launch_bounds__(kE2Block)
k_events_e2(const SgTables tb, const EvArgs a, const int64_t *__restrict__ wave_ev,
            long long w_begin_shared, long long w_end_shared,
            const int64_t *__restrict__ wave_off, int day_index, int slots) {
  constexpr int C = ModelTraits<KIND>::C;
  extern __shared__ __align__(16) int s_state[];
  __shared__ int32_t s_node[kE2Cap], s_dest[kE2Cap], s_n[kE2Cap];
  __shared__ uint8_t s_sel[kE2Cap];
  __shared__ int8_t s_shift[kE2Cap];
  __shared__ long long s_idx[kE2Cap];
  __shared__ double s_prop[kE2Cap];
  __shared__ uint4 s_w[kE2Cap];
  __shared__ long long s_wave[kE2WaveCap + 1];
  __shared__ int16_t s_hv[kE2Cap];  // the wave's events left to the warps
  __shared__ int s_nhv[3];  // see next_wave
  pdl_trigger();
  const int rep = blockIdx.x;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
  if (threadIdx.x < 3) s_nhv[threadIdx.x] = 0;
  int cw = 0;
  const int Nn = tb.n_nodes;
  long long w0 = w_begin_shared, w1 = w_end_shared;
  if (slots > 1) {
    w0 = wave_off[(long long)day_index * slots + rep];
    w1 = wave_off[(long long)day_index * slots + rep + 1];
  }
  if (w0 >= w1) {
    pdl_wait();
    return;
  }
  int *gstate = a.u + (long long)rep * Nn * C;
  int *state = SMEM_STATE ? s_state : gstate;
  bool waited = false;
  // `bad`: this thread met an error; `stop`: the block's verdict, taken at a
  // barrier (__syncthreads_or), so every thread leaves the loops together
  bool bad = false, stop = false;
  const uint64_t seed = ((uint64_t)a.k1 << 32) | a.k0;
  const uint32_t tag = (SG_STREAM_EVENTS << 24) | (uint32_t)(a.rep0 + rep);
  unsigned long long applied = 0;
  long long w = w0;
  long long pos = wave_ev[w0];
  const long long pos_end = wave_ev[w1];
  while (pos < pos_end) {
    // stage the bounds of the next waves, then the events [pos, pend) they
    // hold (at most kE2Cap; a wave may continue into the next chunk)
    const long long wn = min(w1 - w, (long long)kE2WaveCap);
    __syncthreads();
    for (long long i = threadIdx.x; i <= wn; i += blockDim.x) s_wave[i] = wave_ev[w + i];
    __syncthreads();
    const long long pend = min(pos + (long long)kE2Cap, s_wave[wn]);
    for (long long i = threadIdx.x; i < pend - pos; i += blockDim.x) {
      const long long j = pos + i;
      const SgEvent ev = load_event(a.ev.rec + j);
      s_node[i] = ev.node;
      s_dest[i] = ev.dest;
      s_n[i] = ev.n;
      s_sel[i] = ev.select;
      s_shift[i] = ev.shift;
      s_prop[i] = ev.proportion;
      const long long idx = ev.index;
      s_idx[i] = idx;
      const U4 f = philox10(U4{0u, (uint32_t)(unsigned long long)idx,
                               (uint32_t)((unsigned long long)idx >> 32), tag},
                            a.k0, a.k1);
      s_w[i] = make_uint4(f.x, f.y, f.z, f.w);
    }
    if (!waited) {
      // the first chunk is staged: now wait for the day kernel's state
      pdl_wait();
      waited = true;
      if (threadIdx.x == 0 && *(volatile int32_t *)&a.err->code != 0) bad = true;
      if (SMEM_STATE) copy_words(s_state, gstate, Nn * C);
    }
    stop = __syncthreads_or(bad);
    if (stop) break;
    // waves w .. (staged) intersecting [pos, pend)
    long long wi = 0;
    while (wi < wn && s_wave[wi] < pend) {
      const long long lo = max(pos, s_wave[wi]), hi = min(pend, s_wave[wi + 1]);
      for (long long q = lo + threadIdx.x; q < hi; q += blockDim.x) {
        const int i = (int)(q - pos);
        const int src = s_node[i];
        int *un = state + (long long)src * C;
        const uint32_t mask = tb.Emask[s_sel[i]];
        int cur[C];
        long long total = 0;
#pragma unroll
        for (int p = 0; p < C; ++p) {
          cur[p] = un[p];
          if ((mask >> p) & 1u) total += cur[p];
        }
        const long long k = s_n[i] > 0 ? (long long)s_n[i]
                                       : (long long)round(s_prop[i] * (double)total);
        if (k < 0 || k > total) {
          report(a.err, SG_ERR_EVENT_UNDERFLOW, a.rep0 + rep, src, a.day, s_idx[i]);
          bad = true;
          continue;
        }
        if (k >= kUrnWarp) {
          // a large transfer: sampled by a warp after this pass
          s_hv[atomicAdd(&s_nhv[cw], 1)] = (int16_t)i;
          continue;
        }
        int moved[C];
#pragma unroll
        for (int p = 0; p < C; ++p) moved[p] = 0;
        if (k > 0) {
          WordStream ws;
          const uint4 f = s_w[i];
          ws.init_with_first(seed, s_idx[i], a.rep0 + rep, U4{f.x, f.y, f.z, f.w});
          for (long long d = 0; d < k; ++d) {
            uint32_t x = ws.below((uint32_t)(total - d));
            bool taken = false;
#pragma unroll
            for (int p = 0; p < C; ++p) {
              if (taken || !((mask >> p) & 1u)) continue;
              const uint32_t rem = (uint32_t)(cur[p] - moved[p]);
              if (x < rem) {
                ++moved[p];
                taken = true;
              } else {
                x -= rem;
              }
            }
          }
        }
        const int q_sh = s_shift[i];
        int *ud = state + (long long)s_dest[i] * C;
#pragma unroll
        for (int p = 0; p < C; ++p) {
          if (moved[p] == 0) continue;
          un[p] = cur[p] - moved[p];
        }
#pragma unroll
        for (int p = 0; p < C; ++p) {
          if (moved[p] == 0) continue;
          atomicAdd(ud + (q_sh >= 0 ? p + tb.Nsh[q_sh][p] : p), moved[p]);
        }
        ++applied;
      }
      stop = __syncthreads_or(bad);
      if (stop) break;
      const int nhv = next_wave(s_nhv, cw);
      if (nhv > 0) {
        // the wave's large transfers, one warp each: no other event of the
        // wave touches their source nodes, so the order does not matter
        for (int h = warp; h < nhv; h += nwarps) {
          const int i = s_hv[h];
          const int src = s_node[i];
          int *un = state + (long long)src * C;
          const uint32_t mask = tb.Emask[s_sel[i]];
          int cur[C];
          long long total = 0;
#pragma unroll
          for (int p = 0; p < C; ++p) {
            cur[p] = un[p];
            if ((mask >> p) & 1u) total += cur[p];
          }
          const long long k = s_n[i] > 0 ? (long long)s_n[i]
                                         : (long long)round(s_prop[i] * (double)total);
          int moved[C];
          urn_warp<C>(cur, mask, (uint32_t)k, (uint32_t)total, seed, s_idx[i], a.rep0 + rep,
                      moved);
          if (lane == 0) {
            const int q_sh = s_shift[i];
            int *ud = state + (long long)s_dest[i] * C;
#pragma unroll
            for (int p = 0; p < C; ++p)
              if (moved[p] != 0) un[p] = cur[p] - moved[p];
#pragma unroll
            for (int p = 0; p < C; ++p)
              if (moved[p] != 0) atomicAdd(ud + (q_sh >= 0 ? p + tb.Nsh[q_sh][p] : p), moved[p]);
            ++applied;
          }
          __syncwarp();
        }
        __syncthreads();
      }
      if (s_wave[wi + 1] <= pend) ++wi;
      else break;  // the wave continues in the next chunk
    }
    if (stop) break;
    w += wi;
    pos = pend;
  }
  if (!waited) pdl_wait();
  if (SMEM_STATE && waited) {
    __syncthreads();
    copy_words(gstate, s_state, Nn * C);
  }
  if (applied) atomicAdd(&a.cnt->events, applied);
}

// U_sparse / V_sparse entries and prevalence counters of tspan slot 0 (the
// initial state), one thread per (replicate, node).
template <int C, int NV>
__global__ void k_record0(const int32_t *__restrict__ u0, const double *__restrict__ v0, int Nn,
                          int n_rep, int M, const OutDev o) {
  const long long gid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const bool in_range = gid < (long long)Nn * n_rep;
  int u[C];
  double v[NV > 0 ? NV : 1];
#pragma unroll
  for (int p = 0; p < C; ++p) u[p] = 0;
  v[0] = 0.0;
  int rep = 0;
  if (in_range) {
    rep = (int)(gid / Nn);
    const int node = (int)(gid - (long long)rep * Nn);
#pragma unroll
    for (int p = 0; p < C; ++p) u[p] = u0[gid * C + p];
#pragma unroll
    for (int q = 0; q < NV; ++q) v[q] = v0[gid * NV + q];
    record_sparse<C, NV>(o, 0, rep, node, u, v);
  }
  if (o.prev) prevalence_add<C>(o, in_range ? (long long)rep * M : -1, in_range, u);
}

}  // namespace sg
