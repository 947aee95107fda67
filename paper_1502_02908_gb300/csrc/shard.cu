// Exchange kernels of the node-sharded single replicate (sim_shard,
// sim_pack_touched, sim_unpack_touched).
//
// Each rank holds the whole state but runs the stochastic step and the phi update
// (Eqs. (numstep3), (numstep5)) only for its own contiguous node range; every rank
// applies the whole day's event list (Eq. (numstep4)).  Between the two, the herds
// the day's events touch must hold their post-stochastic-step counts on every
// rank: each rank packs those herds' counts, the ranks gather the packs in rank
// order, and each rank takes every touched herd's counts from the pack of the rank
// that owns it.  This is the daily exchange of Sec. 3.4's crossing events, made
// over the touched herds rather than over a split of the event list.
#include "internal.h"

#include <algorithm>

namespace episim {
namespace {

// out [R][Nc][n_t] = counts of the n_t touched herds (plane = r * Nc + c).
__global__ void __launch_bounds__(256) k_pack_touched(const int32_t* __restrict__ counts,
                                                       const int32_t* __restrict__ touched, int n_t, int N,
                                                       int64_t planes, int32_t* __restrict__ out) {
  const int64_t total = planes * n_t;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t plane = i / n_t;
    const int t = (int)(i - plane * n_t);
    out[i] = counts[plane * N + touched[t]];
  }
}

// counts of touched herd v = the pack of v's owner: in [world][R][Nc][n_t];
// bounds [world + 1] (rank k owns [bounds[k], bounds[k+1])); the owner is the
// largest k with bounds[k] <= v, which skips ranks with empty ranges.
__global__ void __launch_bounds__(256) k_unpack_touched(int32_t* __restrict__ counts,
                                                         const int32_t* __restrict__ touched, int n_t, int N,
                                                         int64_t planes, const int32_t* __restrict__ in,
                                                         const int32_t* __restrict__ bounds, int world,
                                                         const int32_t* __restrict__ ids) {
  const int64_t total = planes * n_t;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t plane = i / n_t;
    const int t = (int)(i - plane * n_t);
    const int v = touched[t], id = ids ? ids[v] : v;
    int lo = 0, hi = world - 1;
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (bounds[mid] <= id) lo = mid; else hi = mid - 1;
    }
    counts[plane * N + v] = in[(int64_t)lo * total + i];
  }
}

// Storage order to node order and back: a thread takes one position through the planes
// (grid y of them at a time), so its node is read once.  The scattered side of a plane (a
// few hundred KB) stays in L2, the other streams.
template <bool TO_NODES>
__global__ void __launch_bounds__(256) k_reorder(int32_t* __restrict__ c_out, const int32_t* __restrict__ c_in, int64_t pc,
                                                  double* __restrict__ f_out, const double* __restrict__ f_in, int64_t pf,
                                                  const int32_t* __restrict__ ids, int N) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= N) return;
  const int64_t id = ids[i], to = TO_NODES ? id : i, from = TO_NODES ? i : id;
  for (int64_t p = blockIdx.y; p < pc + pf; p += gridDim.y) {
    if (p < pc) c_out[p * N + to] = c_in[p * N + from];
    else f_out[(p - pc) * N + to] = f_in[(p - pc) * N + from];
  }
}

unsigned grid_for(int64_t total) {
  const int64_t b = (total + 255) / 256;
  return (unsigned)(b < 4096 ? (b > 0 ? b : 1) : 4096);
}

template <bool TO_NODES>
cudaError_t launch_reorder(int32_t* c_out, const int32_t* c_in, int64_t pc, double* f_out, const double* f_in, int64_t pf,
                           const int32_t* ids, int N, cudaStream_t st) {
  if (N <= 0 || pc + pf <= 0) return cudaSuccess;
  const dim3 grid((unsigned)((N + 255) / 256), (unsigned)std::min<int64_t>(pc + pf, 64));
  k_reorder<TO_NODES><<<grid, 256, 0, st>>>(c_out, c_in, pc, f_out, f_in, pf, ids, N);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_to_nodes(int32_t* c_out, const int32_t* c_in, int64_t pc, double* f_out, const double* f_in, int64_t pf,
                            const int32_t* ids, int N, cudaStream_t st) {
  return launch_reorder<true>(c_out, c_in, pc, f_out, f_in, pf, ids, N, st);
}

cudaError_t launch_from_nodes(int32_t* c_out, const int32_t* c_in, int64_t pc, double* f_out, const double* f_in, int64_t pf,
                              const int32_t* ids, int N, cudaStream_t st) {
  return launch_reorder<false>(c_out, c_in, pc, f_out, f_in, pf, ids, N, st);
}

cudaError_t launch_pack_touched(const int32_t* counts, const int32_t* touched, int n_t, int N, int64_t planes,
                                int32_t* out, cudaStream_t st) {
  if (n_t <= 0 || planes <= 0) return cudaSuccess;
  k_pack_touched<<<grid_for(planes * n_t), 256, 0, st>>>(counts, touched, n_t, N, planes, out);
  return cudaGetLastError();
}

cudaError_t launch_unpack_touched(int32_t* counts, const int32_t* touched, int n_t, int N, int64_t planes,
                                  const int32_t* in, const int32_t* bounds, int world, const int32_t* ids,
                                  cudaStream_t st) {
  if (n_t <= 0 || planes <= 0) return cudaSuccess;
  k_unpack_touched<<<grid_for(planes * n_t), 256, 0, st>>>(counts, touched, n_t, N, planes, in, bounds, world, ids);
  return cudaGetLastError();
}

}  // namespace episim
