// Region statistics of the parameter-fitting goal (Sec. 4.3, Eqs. (goal),
// (goalvariance), (goalsigma)): after each day, per replicate i, region j and
// compartment c, the region total x_jc^i = sum over the region's nodes of the
// node's count; accumulated over replicates as exact integers
//   s1[d][j][c] = sum_i x_jc^i,   s2[d][j][c] = sum_i (x_jc^i)^2.
// The goal over days [d0, d0 + n) against a reference trajectory's region totals
// ref[d][j][c] (R = number of trajectories):
//   G^2  = sum_d sum_j sum_c (s1 / R - ref)^2
//   VG^2 = sum_d sum_j sum_c (s2 - s1^2 / R) / (R - 1)
// (the time integral of the paper taken over the daily observations, dt = 1).
#include "internal.h"

#include <algorithm>

namespace episim {

namespace {

constexpr int kRegionThreads = 256;

// One block per (replicate, region): the region's nodes (region-sorted list) are
// summed per compartment, then the block adds the totals and their squares.
__global__ void __launch_bounds__(kRegionThreads) k_region_day(const int32_t* __restrict__ counts,
                                                               const int32_t* __restrict__ reg_nodes,
                                                               const int32_t* __restrict__ reg_off, int N, int R,
                                                               int Nc, int J, int day, unsigned long long* s1,
                                                               unsigned long long* s2) {
  __shared__ long long part[kRegionThreads / 32][6];
  const int r = (int)(blockIdx.x / (unsigned)J), j = (int)(blockIdx.x % (unsigned)J);
  long long acc[6] = {0, 0, 0, 0, 0, 0};
  const int32_t* X = counts + (size_t)r * Nc * N;
  for (int i = reg_off[j] + (int)threadIdx.x; i < reg_off[j + 1]; i += blockDim.x) {
    const int v = reg_nodes[i];
    for (int c = 0; c < Nc; ++c) acc[c] += __ldcg(X + (size_t)c * N + v);
  }
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int c = 0; c < Nc; ++c) {
    long long v = acc[c];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (lane == 0) part[warp][c] = v;
  }
  __syncthreads();
  if (threadIdx.x < (unsigned)Nc) {
    const int c = threadIdx.x;
    long long tot = 0;
    for (int w = 0; w < kRegionThreads / 32; ++w) tot += part[w][c];
    const size_t at = ((size_t)day * J + j) * Nc + c;
    atomicAdd(s1 + at, (unsigned long long)tot);
    atomicAdd(s2 + at, (unsigned long long)(tot * tot));
  }
}

// The same from slabs of consecutive nodes (blockIdx.y the replicate): the counts stream
// in coalesced, one shared-memory add per node and compartment into the block's
// [region][compartment] table -- the low and high 16 bits of a count in tables of their
// own, so that 4,096 nodes of 2^30 animals cannot overflow; the high ones are rarely
// non-zero.  The last block of a replicate turns its totals into s1 and s2 and clears
// them for the next day.  Gathering region by region instead reads a 32-byte sector per
// count: ten national replicates, 21 regions, 19.7 us a launch against 8.1 here (cold caches,
// one GB300), 23.2 -> 21.8 ms for the goal of a year.
template <int NC>
__global__ void __launch_bounds__(kRegionThreads) k_region_slab(const int32_t* __restrict__ counts,
                                                                const int32_t* __restrict__ region_of, int N,
                                                                int J, int day, int slab, unsigned long long* tot,
                                                                unsigned* ticket, unsigned long long* s1,
                                                                unsigned long long* s2) {
  extern __shared__ unsigned tab[];                 // [2][J][Nc]: low, high halves
  __shared__ unsigned last;
  const int r = blockIdx.y, cells = J * NC;
  for (int i = threadIdx.x; i < 2 * cells; i += blockDim.x) tab[i] = 0;
  __syncthreads();
  const int32_t* X = counts + (size_t)r * NC * N;
  const int end = min(N, ((int)blockIdx.x + 1) * slab);
#pragma unroll 2
  for (int v = (int)blockIdx.x * slab + (int)threadIdx.x; v < end; v += kRegionThreads) {
    unsigned* t = tab + region_of[v] * NC;
    unsigned x[NC];
#pragma unroll
    for (int c = 0; c < NC; ++c) x[c] = (unsigned)__ldcg(X + (size_t)c * N + v);
#pragma unroll
    for (int c = 0; c < NC; ++c) {
      if (x[c] & 0xffffu) atomicAdd(t + c, x[c] & 0xffffu);
      if (x[c] >> 16) atomicAdd(t + cells + c, x[c] >> 16);
    }
  }
  __syncthreads();
  unsigned long long* T = tot + (size_t)r * cells;
  for (int i = threadIdx.x; i < cells; i += blockDim.x) {
    const unsigned long long x = (unsigned long long)tab[i] + ((unsigned long long)tab[cells + i] << 16);
    if (x) atomicAdd(T + i, x);
  }
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) last = atomicAdd(ticket + r, 1u) == gridDim.x - 1;
  __syncthreads();
  if (!last) return;
  __threadfence();
  for (int i = threadIdx.x; i < cells; i += blockDim.x) {
    const unsigned long long x = __ldcg(T + i);
    T[i] = 0;
    atomicAdd(s1 + (size_t)day * cells + i, x);
    atomicAdd(s2 + (size_t)day * cells + i, x * x);
  }
  if (threadIdx.x == 0) ticket[r] = 0;
}

// One block: each thread sums its strided terms in order, then a fixed-order
// tree reduction (deterministic).  Differences and variances are formed exactly
// in 128-bit integers before the division.
__global__ void __launch_bounds__(kRegionThreads) k_goal(const unsigned long long* __restrict__ s1,
                                                         const unsigned long long* __restrict__ s2,
                                                         const long long* __restrict__ ref, long long first,
                                                         long long count, int R, double* out) {
  __shared__ double gs[kRegionThreads], vs[kRegionThreads];
  double g = 0.0, v = 0.0;
  for (long long i = threadIdx.x; i < count; i += blockDim.x) {
    const long long a = (long long)s1[first + i], b = (long long)s2[first + i];
    const __int128 diff = (__int128)a - (__int128)R * ref[i];       // R (mean - ref)
    const double d = (double)diff / (double)R;
    g = __dadd_rn(g, __dmul_rn(d, d));
    if (R > 1) {
      const __int128 m2 = (__int128)R * b - (__int128)a * a;         // R (R - 1) sigma^2, exact
      v = __dadd_rn(v, (double)m2 / ((double)R * (double)(R - 1)));
    }
  }
  gs[threadIdx.x] = g;
  vs[threadIdx.x] = v;
  __syncthreads();
  for (int s = kRegionThreads / 2; s > 0; s >>= 1) {
    if (threadIdx.x < (unsigned)s) {
      gs[threadIdx.x] = __dadd_rn(gs[threadIdx.x], gs[threadIdx.x + s]);
      vs[threadIdx.x] = __dadd_rn(vs[threadIdx.x], vs[threadIdx.x + s]);
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) { out[0] = gs[0]; out[1] = vs[0]; }
}

}  // namespace

cudaError_t launch_region_day(const int32_t* counts, const int32_t* reg_nodes, const int32_t* reg_off, int N, int R,
                              int Nc, int J, int day, unsigned long long* s1, unsigned long long* s2,
                              cudaStream_t st) {
  k_region_day<<<(unsigned)((int64_t)R * J), kRegionThreads, 0, st>>>(counts, reg_nodes, reg_off, N, R, Nc, J, day,
                                                                       s1, s2);
  return cudaGetLastError();
}

bool region_slab_fits(int J, int Nc) { return (size_t)J * Nc * 8 <= 32 * 1024; }

cudaError_t launch_region_slab(const int32_t* counts, const int32_t* region_of, int N, int R, int Nc, int J, int day,
                               int sms, unsigned long long* tot, unsigned* ticket, unsigned long long* s1,
                               unsigned long long* s2, cudaStream_t st) {
  // slabs of 256 to 4,096 nodes, about four blocks an SM
  const int64_t want = ((int64_t)N * R + 4 * sms - 1) / (4 * sms);
  const int slab = (int)std::min<int64_t>(4096, std::max<int64_t>(256, (want + 255) / 256 * 256));
  const dim3 grid((unsigned)((N + slab - 1) / slab), (unsigned)R);
  if (Nc == 2) k_region_slab<2><<<grid, kRegionThreads, (size_t)J * 16, st>>>(counts, region_of, N, J, day, slab, tot, ticket, s1, s2);
  else k_region_slab<6><<<grid, kRegionThreads, (size_t)J * 48, st>>>(counts, region_of, N, J, day, slab, tot, ticket, s1, s2);
  return cudaGetLastError();
}

cudaError_t launch_goal(const unsigned long long* s1, const unsigned long long* s2, const long long* ref,
                        long long first, long long count, int R, double* out, cudaStream_t st) {
  k_goal<<<1, kRegionThreads, 0, st>>>(s1, s2, ref, first, count, R, out);
  return cudaGetLastError();
}

}  // namespace episim
