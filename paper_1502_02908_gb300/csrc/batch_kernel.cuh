// Persistent work-stealing kernel (template) for batched and uneven runs: several
// simulations (handles, each with its model, nodes, replicates, horizon, events
// and parameters) advance together in one launch.
//
// Work items, in a fixed global order that every block fetches from one atomic
// counter: for each step s (day day0 + s of every instance still running), first
// the stochastic-step chunks of every (instance, replicate) -- a chunk is
// kBatchSubs blocks' worth of nodes with one thread each, or one large herd per
// warp -- then the event item of every (instance, replicate); after the last
// step, finalisation chunks (phi update and statistics of each instance's last
// day).  A chunk of day d waits until the events of day d-1 of its replicate are
// applied; an event item waits until every chunk of its day is done.
// Dependencies always point to earlier items, and a block fetches an item only
// while it runs, so the earliest unfinished item can always proceed: no
// co-residency assumption is needed.  The items a block fetches only increase,
// so a block decodes each by a galloping search of the step and instance tables
// from its previous item's position.  Waits spin on acquire loads with a bounded
// count (about two seconds); running out sets an error and an abort flag that
// every block checks, and the kernel returns instead of hanging.  State written
// by other blocks is read with L2-coherent loads (see ssa_device.cuh,
// events_device.cuh).
#pragma once
#include "batch.h"
#include "events_device.cuh"
#include "ssa_device.cuh"

namespace episim {

namespace {

__device__ __forceinline__ unsigned ld_acquire(const unsigned* p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

__device__ __forceinline__ int ld_relaxed_int(const int* p) {
  int v;
  asm volatile("ld.relaxed.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

// Waits until *p >= target.  Returns false when the wait ran out or the run was aborted.
__device__ bool wait_at_least(const unsigned* p, unsigned target, const BatchCtl& c) {
  if (ld_acquire(p) >= target) return true;
  for (long long it = 0; it < c.spin_limit; ++it) {
    __nanosleep(128);
    if (ld_acquire(p) >= target) return true;
    if (ld_relaxed_int(c.abort)) return false;
  }
  atomicOr(c.err, kBatchTimeout);
  atomicExch(c.abort, 1);
  return false;
}

// Largest k in [lo, n) with cum[k] <= x, for non-decreasing cum and cum[lo] <= x:
// steps of 1, 2, 4, ... from lo, then a binary search within the last step.
__device__ __forceinline__ int upper_index_from(const long long* cum, int n, int lo, long long x) {
  int step = 1;
  while (lo + step < n && cum[lo + step] <= x) {
    lo += step;
    step <<= 1;
  }
  int hi = min(lo + step, n) - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (cum[mid] <= x) lo = mid; else hi = mid - 1;
  }
  return lo;
}

__device__ __forceinline__ int upper_index(const long long* cum, int n, long long x) {
  // largest k in [0, n) with cum[k] <= x (cum non-decreasing, cum[0] = 0)
  int lo = 0, hi = n - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (cum[mid] <= x) lo = mid; else hi = mid - 1;
  }
  return lo;
}

template <int NA, bool SCORE, int MODE>
__device__ __forceinline__ void run_chunk(const BatchInst& I, int r, int chunk, int day, int prologue) {
  SsaArgs a = I.ssa;
  a.day = day;
  a.prologue = prologue;
  const int wb = (MODE == 0 && !SCORE) ? a.warp_blocks : 0;
  if (MODE == 1 || chunk < wb) { node_day_block<NA, SCORE, MODE>(a, r, chunk); return; }
  // A per-thread chunk is I.subs blocks' worth of nodes, run one after another with
  // no barrier between them: a warp's time is then a sum over I.subs nodes a lane,
  // and the block's closing barrier waits on sums that differ less than single
  // node-days do.
  const int q0 = (chunk - wb) * I.subs;
  for (int j = 0; j < I.subs; ++j) {
    if ((q0 + j) * (int)blockDim.x >= I.n_thread) break;
    node_day_block<NA, SCORE, MODE>(a, r, wb + q0 + j);
  }
}

template <bool SCORE_ANY>
__device__ __forceinline__ void dispatch_chunk(const BatchInst& I, int r, int chunk, int day, int prologue, int mode) {
  if (I.na == 1) {
    if (SCORE_ANY && I.score) { if (mode == 0) run_chunk<1, SCORE_ANY, 0>(I, r, chunk, day, prologue); else run_chunk<1, SCORE_ANY, 1>(I, r, chunk, day, prologue); }
    else { if (mode == 0) run_chunk<1, false, 0>(I, r, chunk, day, prologue); else run_chunk<1, false, 1>(I, r, chunk, day, prologue); }
  } else {
    if (SCORE_ANY && I.score) { if (mode == 0) run_chunk<3, SCORE_ANY, 0>(I, r, chunk, day, prologue); else run_chunk<3, SCORE_ANY, 1>(I, r, chunk, day, prologue); }
    else { if (mode == 0) run_chunk<3, false, 0>(I, r, chunk, day, prologue); else run_chunk<3, false, 1>(I, r, chunk, day, prologue); }
  }
}

// Part `part` of a day's events by owner lists: a component's events are one thread's
// list in input order, so a lane applies it straight to the counts, with no levels, no
// barrier and no staging.  The lists of an owner-computes block go to kBatchEvLanes lanes.
// Bound by the longest list's chain (about 1,200 cycles an event); the staged step takes
// one block through every level of the day: 7,972 herds, 1,747 events a day, one GB300:
// 22 us a day staged, 5 in five parts.
template <int NA>
__device__ __forceinline__ void events_by_lists(const BatchInst& I, int r, int day, int part) {
  const int2 D = __ldg(I.day_df + day);
  EvArgs a = I.evg;
  a.day = day;
  int32_t* X = a.counts + (size_t)r * a.Nc * a.N;
  unsigned applied = 0, clamped = 0, skipped = 0;
  const int sub = threadIdx.x % kBatchEvLanes, per = (int)blockDim.x / kBatchEvLanes;
  for (int b = part * per + (int)threadIdx.x / kBatchEvLanes; b < D.y; b += I.ev_parts * per) {
    const int4 m0 = __ldg(I.df_meta + D.x + b), m1 = __ldg(I.df_meta + D.x + b + 1);
    const int lists = m1.z - m0.z - 1;
    for (int i = sub; i < lists; i += kBatchEvLanes) {
      const int q1 = __ldg(I.df_thr_off + m0.z + i + 1);
      for (int q = __ldg(I.df_thr_off + m0.z + i); q < q1; ++q) {
        int4 rec = __ldg(I.df_rec + m0.x + q);       // slots of the block's touched list
        rec.x = __ldg(I.df_touched + m0.y + rec.x);
        if (rec.y >= 0) rec.y = __ldg(I.df_touched + m0.y + rec.y);
        apply_event<NA>(a, X, r, rec, applied, clamped, skipped);
      }
    }
  }
  applied = __reduce_add_sync(0xffffffffu, applied);
  clamped = __reduce_add_sync(0xffffffffu, clamped);
  skipped = __reduce_add_sync(0xffffffffu, skipped);
  if ((threadIdx.x & 31) == 0) {
    unsigned long long* c = a.ctr + (size_t)r * 4;
    if (applied) atomicAdd(c + 1, (unsigned long long)applied);
    if (clamped) atomicAdd(c + 2, (unsigned long long)clamped);
    if (skipped) atomicAdd(c + 3, (unsigned long long)skipped);
  }
}

template <bool LISTS>
__device__ __forceinline__ void dispatch_events(const BatchInst& I, int r, int day, int part, unsigned char* smem,
                                                int smem_cap) {
  if (!I.has_events) return;
  const int dl0 = __ldg(I.evg.day_lvl + day), dl1 = __ldg(I.evg.day_lvl + day + 1);
  if (dl1 <= dl0) return;
  if (LISTS && I.by_lists && __ldg(&I.day_df[day].y) > 0) {
    if (I.na == 1) events_by_lists<1>(I, r, day, part); else events_by_lists<3>(I, r, day, part);
    return;
  }
  if (part > 0) return;
  const int need = __ldg(I.day_smem + day);
  if (need > 0 && need <= smem_cap) {
    EvSmemArgs a = I.evs;
    a.day = day;
    a.smem_bytes = need;
    if (I.na == 1) events_block_smem<1>(a, r, smem); else events_block_smem<3>(a, r, smem);
  } else {
    EvArgs a = I.evg;
    a.day = day;
    if (I.na == 1) events_block_global<1>(a, r); else events_block_global<3>(a, r);
  }
}

// THREADS threads a block, MINB blocks an SM (the register budget), whether any
// instance computes the score and whether any takes its events by lists (either step is
// compiled in only then: the lists' registers cost the batched national run 8 %).
template <int THREADS, int MINB, bool SCORE_ANY, bool LISTS>
__global__ void __launch_bounds__(THREADS, MINB) k_batch(BatchCtl c) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ long long s_item;
  __shared__ int s_go;   // written by thread 0 only before the loop-top barrier
  __shared__ int s_ok;   // the item's dependency wait succeeded (its own flag: s_go
                         // may still be being read when the wait's result lands)
  __shared__ int s_hs, s_hk, s_hkind;   // the previous item's step, instance and kind (0 chunk, 1 events)
  if (threadIdx.x == 0) { s_hs = 0; s_hk = 0; s_hkind = -1; }   // read after the loop's first barrier
  for (;;) {
    if (threadIdx.x == 0) {
      s_item = (long long)atomicAdd(c.next, 1ull);
      s_go = (s_item < c.total) && !ld_relaxed_int(c.abort);
    }
    __syncthreads();
    const long long t = s_item;
    if (!s_go) break;
    if (t < c.total_main) {
      const int hs = s_hs, hk = s_hk, hkind = s_hkind;
      const int s = upper_index_from(c.step_off, c.n_steps, hs, t);
      const long long local = t - c.step_off[s];
      const int act = c.active[s];
      const long long nA = c.cumA[act];
      int k, r, chunk = 0;                            // chunk: of the stochastic step, or part of the events
      const bool is_ssa = local < nA;
      if (is_ssa) {
        k = upper_index_from(c.cumA, act, (hs == s && hkind == 0) ? hk : 0, local);
        const long long w = local - c.cumA[k];
        const BatchInst& I0 = c.inst[k];
        r = (int)(w / I0.bpr);
        chunk = (int)(w - (long long)r * I0.bpr);
      } else {
        k = upper_index_from(c.cumB, act, (hs == s && hkind == 1) ? hk : 0, local - nA);
        const long long w = local - nA - c.cumB[k];
        const int parts = c.inst[k].ev_parts;
        r = (int)(w / parts);
        chunk = (int)(w - (long long)r * parts);
      }
      const BatchInst& I = c.inst[k];
      const int day = I.day0 + s;
      if (threadIdx.x == 0) s_ok = is_ssa ? wait_at_least(I.ev_done + r, 1u + (unsigned)(s * I.ev_parts), c)
                                          : wait_at_least(I.ssa_done + r, (unsigned)((s + 1) * I.bpr), c);
      __syncthreads();
      if (s_ok) {
        if (is_ssa) dispatch_chunk<SCORE_ANY>(I, r, chunk, day, s > 0, 0);
        else dispatch_events<LISTS>(I, r, day, chunk, smem, c.smem_cap);
      }
      __syncthreads();
      if (threadIdx.x == 0) { s_hs = s; s_hk = k; s_hkind = is_ssa ? 0 : 1; }   // read after the next barrier
      if (threadIdx.x == 0 && s_ok) {
        __threadfence();
        atomicAdd((is_ssa ? I.ssa_done : I.ev_done) + r, 1u);
      }
    } else {
      const long long local = t - c.total_main;
      const int k = upper_index(c.cumF, c.n_inst, local);
      const BatchInst& I = c.inst[k];
      const long long w = local - c.cumF[k];
      const int r = (int)(w / I.tbpr), chunk = (int)(w - (long long)r * I.tbpr);
      const int last = I.day0 + I.ndays - 1;
      if (threadIdx.x == 0) s_ok = wait_at_least(I.ev_done + r, 1u + (unsigned)(I.ndays * I.ev_parts), c);
      __syncthreads();
      if (s_ok) dispatch_chunk<SCORE_ANY>(I, r, chunk, last, 1, 1);
    }
    __syncthreads();
  }
}

}  // namespace

// The kernel of one block shape with the score step compiled in or not, and with the list
// events; each is instantiated in a translation unit of its own (batch_shape_*.cu,
// batch_lists_*.cu).
template <int THREADS, int MINB>
BatchKernel batch_kernel_of(BatchForm f) {
  return f == BatchForm::kScore ? (BatchKernel)k_batch<THREADS, MINB, true, false>
                                : (BatchKernel)k_batch<THREADS, MINB, false, false>;
}
template <int THREADS, int MINB>
BatchKernel batch_lists_of() {
  return (BatchKernel)k_batch<THREADS, MINB, false, true>;
}

}  // namespace episim
