// Descriptors of the persistent batch kernel (batch.cu), filled by host.cpp.
#pragma once
#include "internal.h"

namespace episim {

// Block shapes of the persistent kernel: threads a block x blocks an SM (the
// register budget).  A stochastic-step chunk is one block's worth of nodes (one a
// thread) or of large herds (one a warp), so the shape also sets the chunk size.
enum class BatchShape { k256x1, k256x2, k128x4 };
constexpr int batch_threads(BatchShape s) { return s == BatchShape::k128x4 ? 128 : 256; }
constexpr int batch_min_blocks(BatchShape s) {
  return s == BatchShape::k256x2 ? 2 : s == BatchShape::k128x4 ? 4 : 1;
}
constexpr int kBatchTimeout = 2;      // error bit: a bounded wait ran out
constexpr int kBatchEvLanes = 4;      // lanes an owner-computes block's lists are dealt to
constexpr int kBatchEvLongest = 32;   // longest owner list the lanes take
constexpr int kBatchSubs = 4;         // most blocks' worth of per-thread nodes in a chunk

struct BatchInst {
  SsaArgs ssa;            // node order / warp split set for one block's chunks
  EvSmemArgs evs;
  EvArgs evg;
  const int32_t* day_smem;  // [max_days] shared memory of the staged event step (0: global variant)
  // owner lists of the owner-computes form (EvDfArgs), for the event items in parts
  const int4* df_rec;
  const int32_t* df_thr_off;
  const int32_t* df_touched;
  const int4* df_meta;
  const int2* day_df;       // [max_days] {first block, blocks; 0 where a day's lists do not suit}
  int32_t by_lists;         // whether days with lists take them
  int32_t ev_parts;         // event items per replicate and day
  int32_t na, score, has_events;
  int32_t bpr;            // stochastic-step chunks per replicate
  int32_t subs;           // blocks' worth of per-thread nodes in one chunk
  int32_t n_thread;       // nodes on the per-thread path
  int32_t tbpr;           // finalisation chunks per replicate
  int32_t day0, ndays;
  unsigned* ssa_done;     // [R] chunks completed in this run
  unsigned* ev_done;      // [R] 1 + event items completed in this run
};

struct BatchCtl {
  const BatchInst* inst;  // [n_inst], longest horizon first
  const long long* cumA;  // [n_inst + 1] prefix sums of R * bpr
  const long long* cumB;  // [n_inst + 1] prefix sums of R * ev_parts
  const long long* cumF;  // [n_inst + 1] prefix sums of R * tbpr
  const long long* step_off;  // [n_steps + 1] first item of each step
  const int32_t* active;  // [n_steps] instances still running at each step (a prefix)
  unsigned long long* next;
  int* abort;
  int* err;
  long long total_main, total;
  long long spin_limit;
  int n_inst, n_steps;
  int smem_cap;
};

// What is compiled into the kernel beside the common steps; with any score instance, and
// in blocks of 128 threads, the events are staged.
enum class BatchForm { kPlain, kScore, kLists };
using BatchKernel = void (*)(BatchCtl);
BatchKernel batch_kernel_256x1(BatchForm f);
BatchKernel batch_kernel_256x2(BatchForm f);
BatchKernel batch_kernel_128x4(BatchForm f);
BatchKernel batch_lists_256x1();
BatchKernel batch_lists_256x2();

cudaError_t launch_batch(const BatchCtl& c, BatchShape s, BatchForm f, int grid, cudaStream_t st);
cudaError_t batch_occupancy(BatchShape s, BatchForm f, int smem_bytes, int* blocks_per_sm);

}  // namespace episim
