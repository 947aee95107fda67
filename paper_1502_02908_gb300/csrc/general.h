// Internal interfaces of the general compartment model (include/episim_general.h)
// between its host side (general_host.cpp) and its kernels (general.cu).
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

namespace episim {

constexpr int kGenMaxComp = 16, kGenMaxTrans = 32, kGenMaxCont = 4, kGenMaxSelect = 32, kGenMaxShift = 32;
constexpr int kGenNoShift = kGenMaxShift;  // shift row of zero offsets
constexpr int kGenThreads = 128;           // threads per block of every general-model kernel
enum { kGenYPostEvent = 0, kGenYPreEvent = 1, kGenYMidpoint = 2 };

// The model as the kernels read it; every block copies it into shared memory.
struct alignas(16) GenModelDev {
  int32_t nc, nt, ny, y_source;
  int32_t fa[kGenMaxTrans], fb[kGenMaxTrans], fy[kGenMaxTrans];
  uint32_t pop[kGenMaxTrans];
  uint32_t dep[kGenMaxTrans];               // bit j of dep[n]: firing n can change rate j
  int32_t chg_off[kGenMaxTrans + 1];        // change list of transition n: chg[chg_off[n] .. chg_off[n+1])
  int32_t pad0[3];
  uint32_t chg[kGenMaxComp * kGenMaxTrans]; // (delta << 8) | compartment, delta signed
  uint32_t num[kGenMaxCont], den[kGenMaxCont];
  uint32_t select[kGenMaxSelect];
  int8_t shift[kGenMaxShift + 1][kGenMaxComp];  // row kGenNoShift is all zero
  int32_t pad1[4];
};
static_assert(sizeof(GenModelDev) % 16 == 0, "GenModelDev is copied as int4");

// Per-replicate constants.
struct alignas(16) GenRepParams {
  double rate[kGenMaxTrans];
  double alpha[kGenMaxCont];
  double beta[kGenMaxCont][4];
  double eps[kGenMaxCont];
};
static_assert(sizeof(GenRepParams) % 16 == 0, "GenRepParams is copied as int4");

struct GenSsaArgs {
  int32_t* counts;              // [R][Nc][N]
  double* y;                    // [R][Ny][N]
  double* mid;                  // midpoint variant: [R][Ny][2][N] sums U_n, D_n (else NULL)
  const GenModelDev* model;
  const GenRepParams* params;   // [R]
  const int32_t* order;         // node order (largest initial population first)
  unsigned long long* ctr;      // [R][4]
  uint64_t seed;
  int32_t rep_base, N, R, day;
  int32_t n_big;                // leading nodes of the order simulated one per warp
  int32_t n_mid;                // next nodes of the order, four per warp (8-lane segments)
  int32_t warp_blocks;          // binary64 methods: blocks holding the warp nodes (set by the launcher)
  int32_t group_blocks;         // ... the group nodes
  int32_t prologue;             // 1: first apply day - 1's continuous update (post-event or midpoint)
  uint64_t clock_margin;        // Q62 margin of the binary32 clock (0: binary64 methods only)
  float margin_f;               // the same as binary32
  // Change tables, back to back (tab16 16-byte words): [dyn_rows][L] floats, what transition
  // n adds to row r; the thread method's [nt] {row0 | row1 << 16, change0 | change1 << 16,
  // first, end of further changes}; [nt][pk_words] words of four rows' change + 1 a byte;
  // the further {row, change} pairs (rows in elements of a thread's column).
  const float4* tab;
  int32_t tab16;
  int32_t pk_words;             // words of the byte table (0: a change beyond -1..1, or too many rows)
  int32_t nt, L;                // transitions; the power of two the kernel is unrolled for
  int32_t resident_blocks;      // blocks the device holds at once
  int32_t xrows;                // rows of a thread's column: counts, populations, ones, scratch
  int32_t npop, dyn_rows;       // populations; counts and populations a firing can change (these come first)
  uint32_t pops[kGenMaxTrans];  // the distinct population masks
  int32_t fa[kGenMaxTrans], fb[kGenMaxTrans], pr[kGenMaxTrans], fy[kGenMaxTrans];  // rows a rate reads (-1: none)
};

// Event record, 16 bytes: {node, dest, count, kind | select << 8 | shift row << 16}.
struct GenEvArgs {
  int32_t* counts;
  const int4* rec;              // records grouped by (day, component), input order inside
  const int32_t* comp_ev;       // their positions in the day-stable order (Philox counter word 0)
  const int32_t* comp_off;      // [n_components + 1]
  int32_t comp0, ncomp;         // the day's components
  const GenModelDev* model;
  unsigned long long* ctr;
  int32_t* err;                 // bit 0: an event asked for absent animals (ERROR policy)
  uint64_t seed;
  int32_t rep_base, N, R, day, underflow_error;
};

struct GenContArgs {
  int32_t* counts;
  double* y;
  const double* mid;
  const GenModelDev* model;
  const GenRepParams* params;
  int32_t N, R, day;
};

int gen_unroll(int nt);
// Raises the shared-memory limits of the stochastic-step kernels to the device's; the blocks an
// SM holds of this model's.
cudaError_t gen_ssa_prepare(int nc, int nt, int L, int tab16, int xrows, int* blocks_per_sm);
cudaError_t launch_gen_ssa(GenSsaArgs a, int nt, int nc, cudaStream_t st);
cudaError_t launch_gen_events(const GenEvArgs& a, int nc, cudaStream_t st);
cudaError_t launch_gen_cont(const GenContArgs& a, cudaStream_t st);

}  // namespace episim
