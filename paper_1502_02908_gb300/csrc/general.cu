// Kernels of the general compartment model (Secs. 2.1-2.2, 3.1-3.3): the
// stochastic step (direct method per node with a sparse dependency graph), the
// event step (one thread per component of the day's transfer graph) and the
// continuous update (Eqs. (numstep5) and (numstep2)).
//
// Arithmetic: rates, a0, thresholds, tau and the continuous update are binary64
// with the operation order of include/episim_general.h (no contraction; the
// build passes -fmad=false); -log(u) is the exact fixed-point logarithm of the
// SISe kernels; comparisons of non-negative doubles compare bit patterns.
#include "../../include/episim_general.h"
#include "devmath.cuh"
#include "general.h"
#include "softdiv.cuh"
#include "ssa_device.cuh"   // the binary32 helpers of the speculative clock

#include <algorithm>

namespace episim {

namespace {

__device__ __forceinline__ void copy16(void* dst, const void* src, int n16) {
  int4* d = reinterpret_cast<int4*>(dst);
  const int4* s = reinterpret_cast<const int4*>(src);
  for (int i = threadIdx.x; i < n16; i += blockDim.x) d[i] = __ldg(s + i);
}

// Exact binary64 of 0 <= n < 2^53 on the integer pipe.
__device__ __forceinline__ double u2d_exact(long long n) {
  if (n <= 0) return 0.0;
  const uint64_t u = (uint64_t)n;
  const int top = 63 - __clzll(u);
  const uint64_t mant = (u << (52 - top)) & ((1ull << 52) - 1);
  return bits_to_double(((uint64_t)(1023 + top) << 52) | mant);
}

__device__ __forceinline__ long long mask_sum(const int32_t* x, int stride, uint32_t mask, int nc) {
  long long s = 0;
  for (int c = 0; c < nc; ++c)
    if (mask >> c & 1u) s += x[c * stride];
  return s;
}

// a_j = k_j [* y_q] [* x_a] [* x_b] [/ P], left to right (IEEE products; the
// quotient by the integer-pipe division, bit-identical to IEEE).
__device__ __forceinline__ double gen_rate(const GenModelDev& m, const GenRepParams& p, const int32_t* x, int stride,
                                        const double* y, int j) {
  double a = p.rate[j];
  const int q = m.fy[j], fa = m.fa[j], fb = m.fb[j];
  const uint32_t pm = m.pop[j];
  if (q >= 0) a = __dmul_rn(a, y[q]);
  if (fa >= 0) a = __dmul_rn(a, i2d_exact(x[fa * stride]));
  if (fb >= 0) a = __dmul_rn(a, i2d_exact(x[fb * stride]));
  if (pm) {
    const long long P = mask_sum(x, stride, pm, m.nc);
    a = (P > 0 && pos(a)) ? div_pos(a, u2d_exact(P)) : 0.0;
  }
  return a;
}

__device__ __forceinline__ double gen_y_next(const GenModelDev& m, const GenRepParams& p, int q, int day,
                                             double y, double U, double D) {
  const double omb = __dsub_rn(1.0, p.beta[q][season_of(day)]);
  double mid;
  if (m.den[q] == 0u) mid = __dmul_rn(p.alpha[q], U);
  else {
    const double aU = __dmul_rn(p.alpha[q], U);
    mid = D > 0.0 && pos(aU) ? div_pos(aU, D) : 0.0;
  }
  return __dadd_rn(__dadd_rn(__dmul_rn(y, omb), mid), p.eps[q]);
}

// Per-thread rate storage in shared memory: rate j of the thread at a[j * stride],
// its left-to-right partial sum at P[j * stride] (rolled loops keep the kernel
// small enough for the instruction cache).
struct RateRow {
  double* a;
  double* P;
  int stride;
};

// P_j = P_{j-1} + a_j for j >= j0 (P_0 = a_0, which equals 0 + a_0 for a_0 >= 0);
// returns a0 = P_{nt-1}.
__device__ __forceinline__ double prefix_from(const RateRow& R, int nt, int j0) {
  double run = j0 > 0 ? R.P[(j0 - 1) * R.stride] : 0.0;
  for (int j = j0; j < nt; ++j) {
    run = j == 0 ? R.a[0] : __dadd_rn(run, R.a[j * R.stride]);
    R.P[j * R.stride] = run;
  }
  return nt > 0 ? R.P[(nt - 1) * R.stride] : 0.0;
}

// Eq. (sampling2): the first j with a_j > 0 and r <= P_j, else the last j with a_j > 0.
__device__ __forceinline__ int select_transition(const RateRow& R, int nt, double r) {
  int last = -1;
  for (int j = 0; j < nt; ++j)
    if (pos(R.a[j * R.stride])) {
      last = j;
      if (le_nonneg(r, R.P[j * R.stride])) return j;
    }
  return last;
}

__device__ __forceinline__ void apply_changes(const GenModelDev& m, int32_t* x, int stride, int n, int times) {
  for (int q = m.chg_off[n]; q < m.chg_off[n + 1]; ++q) {
    const uint32_t c = m.chg[q];
    x[(c & 0xffu) * stride] += times * ((int32_t)c >> 8);
  }
}

// Direct method of one node-day by one thread (Eqs. (sampling), (sampling2));
// x is the node's counts in shared memory (stride = threads per block).  After a
// firing only the rates of its dependency graph are recomputed, and the partial
// sums from the first of them on.
__device__ __forceinline__ uint32_t gen_node_day(const GenModelDev& m, const GenRepParams& p, int32_t* x,
                                                 int stride, const RateRow& R, const double* y, uint32_t v,
                                                 uint32_t day, uint32_t rep, uint32_t k0, uint32_t k1) {
  const int nt = m.nt;
  for (int j = 0; j < nt; ++j) R.a[j * R.stride] = gen_rate(m, p, x, stride, y, j);
  double a0 = prefix_from(R, nt, 0);
  double t = 0.0;
  uint32_t fired = 0;
  for (uint32_t k = 0; pos(a0); ++k) {
    const uint4 w = philox10(make_uint4(v, day, k, rep), k0, k1);
    const double E = neglog_u((((uint64_t)w.y << 32) | w.x) >> 12);
    const double u2 = uniform_open(w.z, w.w);
    const double tn = __dadd_rn(t, div_pos(E, a0));
    if (le_nonneg(1.0, tn)) break;
    t = tn;
    const int chosen = select_transition(R, nt, __dmul_rn(a0, u2));
    apply_changes(m, x, stride, chosen, 1);
    uint32_t dm = m.dep[chosen];
    const int j0 = dm ? __ffs(dm) - 1 : nt;
    while (dm) {
      const int j = __ffs(dm) - 1;
      dm &= dm - 1u;
      R.a[j * R.stride] = gen_rate(m, p, x, stride, y, j);
    }
    a0 = prefix_from(R, nt, j0);
    ++fired;
  }
  return fired;
}

// Direct method of one node-day by a segment of SEG lanes (a whole warp, SEG =
// 32, or a quarter, SEG = 8, four nodes to a warp), SEG draws per round.  Lane l
// of the segment takes draw k + l.  Its state is the round's base state plus the
// transitions the segment's lanes before it choose; the choices are found by a
// fixed-point iteration (each lane chooses at the state the current choices of
// the lanes before it imply; lane 0's choice is final after one pass, and each
// pass fixes at least one more lane, so the choices settle within SEG passes).
// The clock then runs over the segment's lanes in draw order with the binary64
// sums of the sequential method, so the result is that method's.  Every lane of
// the warp takes part in its collectives; lanes of a segment without a node
// (live = false) only vote.  xl: this lane's counts (shared memory, stride as in
// the thread method); base: the segment's counts at the start of the round;
// ctau, cch: the segment's SEG clock increments and choices; sl, sb: the lane's
// index in its segment and the segment's first lane in the warp.
template <int SEG>
__device__ __forceinline__ uint32_t gen_seg_node_day(const GenModelDev& m, const GenRepParams& p, int32_t* xl,
                                                     int32_t* base, int stride, const RateRow& R, double* ctau,
                                                     int32_t* cch, const double* y, uint32_t v, uint32_t day,
                                                     uint32_t rep, uint32_t k0, uint32_t k1, int sl, int sb,
                                                     bool live) {
  const int nt = m.nt, nc = m.nc;
  const unsigned full = 0xffffffffu;
  const unsigned seg = SEG == 32 ? full : (((1u << SEG) - 1u) << sb);
  const unsigned below = ((1u << sl) - 1u) << sb;
  live = live && nt > 0;
  double t = 0.0;
  uint32_t fired = 0;
  for (uint32_t kb = 0; __any_sync(full, live); kb += SEG) {
    double E = 0.0, u2 = 0.0;
    if (live) {
      const uint4 w = philox10(make_uint4(v, day, kb + (uint32_t)sl, rep), k0, k1);
      E = neglog_u((((uint64_t)w.y << 32) | w.x) >> 12);
      u2 = uniform_open(w.z, w.w);
    }
    int choice = -1;
    double tau = 0.0;
    for (int pass = 0; pass <= SEG; ++pass) {
      if (live)
        for (int c = 0; c < nc; ++c) xl[c * stride] = base[c];
      for (int j = 0; j < nt; ++j) {
        const int cnt = __popc(__ballot_sync(full, live && choice == j) & below);
        if (cnt) apply_changes(m, xl, stride, j, cnt);
      }
      int next = -1;
      if (live) {
        for (int j = 0; j < nt; ++j) R.a[j * R.stride] = gen_rate(m, p, xl, stride, y, j);
        const double a0 = prefix_from(R, nt, 0);
        if (pos(a0)) {
          next = select_transition(R, nt, __dmul_rn(a0, u2));
          tau = div_pos(E, a0);
        }
      }
      const bool changed = __any_sync(full, live && next != choice);
      choice = next;
      if (!changed) break;
    }
    if (live) {
      ctau[sl] = tau;
      cch[sl] = choice;
    }
    __syncwarp();
    // clock over the segment's lanes in draw order (every lane of it runs the same sums)
    int stop = SEG;
    if (live)
      for (int l = 0; l < SEG; ++l) {
        if (cch[l] < 0) { stop = l; break; }
        const double tn = __dadd_rn(t, ctau[l]);
        if (le_nonneg(1.0, tn)) { stop = l; break; }
        t = tn;
      }
    const unsigned fired_lanes = stop == SEG ? seg : (((1u << stop) - 1u) << sb);
    for (int j = 0; j < nt; ++j) {
      const int cnt = __popc(__ballot_sync(full, live && choice == j) & fired_lanes);
      if (cnt && live && sl == 0) apply_changes(m, base, 1, j, cnt);
    }
    __syncwarp();
    if (live) {
      fired += (uint32_t)stop;
      if (stop < SEG) live = false;
    }
  }
  return fired;
}

constexpr int kGenSeg = 8;                          // lanes per node of the group method
constexpr int kGenWarps = kGenThreads / 32;
constexpr int kGenEventWarps = 8192;                // event step: a warp per component up to this many
constexpr int kGenSmall = 4;                         // event step: compartments that stay in registers

// ---------------------------------------------------------------------------
// Binary32 methods.  With u = 2^-24, nt <= 32, every constant k_j y_q 0 or within
// [2^-100, 2^60] and counts and populations below 2^22 (exact in binary32): a
// binary32 rate (the constant truncated, 2u; at most two products, one reciprocal
// of 1 ulp and its product) is within 8u of the binary64 rate, and never 0 unless
// that rate is 0; a sum of non-negative rates adds at most the depth of its
// addition tree.  A selection is taken in binary32 only when r~ and every threshold
// it is compared with are further apart than their bounds, else the exact binary64
// rule decides that draw; a clock decision inside the margin hands the node-day
// back to the binary64 method.  The results are the specification's, bit for bit.
// A positive constant below 2^-100 (a variable that decayed for years) is taken as
// 2^-100: its rate is then too large by at most 2^-56, all of them by 2^-51.  For the
// clock that is at most 2u of any a0~ from 2^-28 on (one clamped rate: u / 16); below that
// no draw is a certain continue, while a certain stop only becomes more certain with the
// true, smaller a0.  For a selection it is an absolute error of 2^-51 in every threshold
// and in r~, so a selection is decisive only from 2^-49 on, besides the relative bound.
constexpr uint32_t kGenSpecMaxSteps = 1u << 18;
constexpr float kGenSmallA0 = 3.7252903e-9f;                  // 2^-28
constexpr float kGenBigCount = 4194304.0f;                    // 2^22

// binary32 constant k_j y_q of a transition; false when outside the bounds above.
__device__ __forceinline__ bool gen_const_f32(double k, bool has_y, double y, float& c) {
  const double ky = has_y ? __dmul_rn(k, y) : k;
  const int e = (int)(double_bits(ky) >> 52) - 1023;
  c = !pos(ky) ? 0.0f : (e < -100 ? 7.8886091e-31f : trunc_to_f32(ky));
  if (has_y && !pos(y) && double_bits(y) != 0ull) return false;   // negative or -0: exact method
  return !pos(ky) || e < 60;
}

// The exact rule of Eq. (sampling2) for state x and uniform u2, in two passes of
// binary64 rates (a0 first, then the running sums): the transition chosen.
__device__ __forceinline__ int gen_exact_choice(const GenModelDev& m, const GenRepParams& p, const int32_t* x,
                                                int stride, const double* y, double u2) {
  const int nt = m.nt;
  double a0 = 0.0;
  for (int j = 0; j < nt; ++j) {
    const double aj = gen_rate(m, p, x, stride, y, j);
    a0 = j == 0 ? aj : __dadd_rn(a0, aj);
  }
  const double r = __dmul_rn(a0, u2);
  double run = 0.0;
  int last = -1;
  for (int j = 0; j < nt; ++j) {
    const double aj = gen_rate(m, p, x, stride, y, j);
    run = j == 0 ? aj : __dadd_rn(run, aj);
    if (pos(aj)) {
      last = j;
      if (le_nonneg(r, run)) return j;
    }
  }
  return last;
}

// A thread's column of shared memory (stride kGenThreads): its node's counts, the
// model's distinct populations (those a firing can change first), a row of ones and a
// scratch row, as binary32.  The column is about to be read as the other of int32 and
// float:
__device__ __forceinline__ void column_retyped() { asm volatile("" ::: "memory"); }

__device__ __forceinline__ void column_to_int(float* xf, int nc) {
  int32_t* xi = reinterpret_cast<int32_t*>(xf);
  for (int c = 0; c < nc; ++c) {
    const int32_t x = (int32_t)xf[c * kGenThreads];
    column_retyped();
    xi[c * kGenThreads] = x;
  }
}

__device__ __forceinline__ void column_to_float(float* xf, int nc) {
  const int32_t* xi = reinterpret_cast<const int32_t*>(xf);
  for (int c = 0; c < nc; ++c) {
    const int32_t x = xi[c * kGenThreads];
    column_retyped();
    xf[c * kGenThreads] = __int2float_rn(x);
  }
  column_retyped();
}

// Rates at the column's state, as left-to-right partial sums P (within (nt + 8)u);
// returns a0.  The rows a rate reads are kernel arguments (uniform), its constants
// registers, so every rate is recomputed without divergence: about eight instructions
// each.
template <int L>
__device__ __forceinline__ float gen_sums_f32(const GenSsaArgs& a, const float (&kyf)[L], const float* xf,
                                              float (&P)[L]) {
  float a0 = 0.0f;
#pragma unroll
  for (int j = 0; j < L; ++j) {
    if (j < a.nt) {
      float r = __fmul_rn(kyf[j], xf[a.fa[j]]);
      if (a.fb[j] >= 0) r = __fmul_rn(r, xf[a.fb[j]]);
      if (a.pr[j] >= 0) {
        const float pop = xf[a.pr[j]];
        r = pop > 0.0f ? __fmul_rn(r, rcp_approx(pop)) : 0.0f;
      }
      a0 = __fadd_rn(a0, r);
    }
    P[j] = a0;
  }
  return a0;
}

// The transition r = a0 u2 fires: the number of thresholds below r (zero-width
// intervals, from zero rates, are skipped), -1 unless r~ (within (nt + 26)u and 2^-51) is
// at least 2^-17 r~ + 2^-49 from every threshold: 2^-17 = 128u, more than 2 nt + 34 <= 98.
template <int L>
__device__ __forceinline__ int gen_select_f32(int nt, const float (&P)[L], float r) {
  float gap = r;
  int n = 0;
#pragma unroll
  for (int j = 0; j < L; ++j)
    if (j < nt) {
      const float e = __fsub_rn(r, P[j]);
      gap = fminf(gap, fabsf(e));
      n += e > 0.0f ? 1 : 0;
    }
  return gap < __fmaf_rn(r, 7.6293945e-6f, 1.7763568e-15f) || n >= nt ? -1 : n;
}

// The thread method: one node per thread.  A firing n applies chg[n] = two (row,
// change) pairs, further ones from more[].  About 100 instructions and 350 cycles a
// step for six transitions.  The clock (as in ssa_node_day_spec) is within (nt + 35)u t
// plus 2^-22 sum(1 / a0~) of the binary64 chain.  Returns the transitions fired, or -1
// for the caller to rerun the node-day.
template <int L>
__device__ __forceinline__ int32_t gen_thread_node_day(const GenSsaArgs& a, const GenModelDev& m,
                                                       const GenRepParams& p, const int4* chg, const int2* more,
                                                       const float (&kyf)[L], float* xf, const double* y, uint32_t v,
                                                       uint32_t rep, uint32_t k0, uint32_t k1, float margin) {
  const int nt = a.nt;
  float hi = 2.0f, lo = 0.0f, mm = margin, nl, u2f;
  uint4 w = philox10(make_uint4(v, (uint32_t)a.day, 0u, rep), k0, k1);
  draw_f32(w, nl, u2f);
  for (uint32_t k = 0;; ++k) {
    float P[L];
    const float a0 = gen_sums_f32<L>(a, kyf, xf, P);
    const uint4 wn = philox10(make_uint4(v, (uint32_t)a.day, k + 1u, rep), k0, k1);
    const float q = rcp_approx(a0);
    const float tau = __fmul_rn(nl, __fmul_rn(q, 0.693147182f));
    const float hn = __fadd_rn(hi, tau);
    lo = __fadd_rn(lo, __fsub_rn(tau, __fsub_rn(hn, hi)));
    hi = hn;
    mm = __fmaf_rn(q, 2.5e-7f, mm);
    const float d = __fadd_rn(__fsub_rn(hi, 3.0f), lo);
    if (!(a0 > 0.0f) || d > -mm || k >= kGenSpecMaxSteps) return (!(a0 > 0.0f) || d >= mm) ? (int32_t)k : -1;
    int n = gen_select_f32<L>(nt, P, __fmul_rn(a0, u2f));
    if (n < 0) {
      column_to_int(xf, m.nc);
      n = gen_exact_choice(m, p, reinterpret_cast<const int32_t*>(xf), kGenThreads, y, uniform_open(w.z, w.w));
      column_to_float(xf, m.nc);
    }
    const int4 e = chg[n];
    const float x0 = __fadd_rn(xf[e.x & 0xffff], (float)(int16_t)(e.y & 0xffff));
    const float x1 = __fadd_rn(xf[e.x >> 16], (float)(e.y >> 16));
    xf[e.x & 0xffff] = x0;
    xf[e.x >> 16] = x1;
    bool over = fmaxf(x0, x1) >= kGenBigCount;
    for (int i = e.z; i < e.w; ++i) {
      const int2 c = more[i];
      const float x = __fadd_rn(xf[c.x], (float)c.y);
      xf[c.x] = x;
      over = over || x >= kGenBigCount;
    }
    if (over) return -1;
    if ((k & 63u) == 63u) {
      const float h = __fadd_rn(hi, lo);
      lo = __fsub_rn(lo, __fsub_rn(h, hi));
      hi = h;
    }
    w = wn;
    draw_f32(w, nl, u2f);
  }
}

// The segment method in binary32: SEG lanes per node, SEG draws a round, decided by the
// fixed-point iteration of gen_seg_node_day.  A pass counts each transition's firings
// below the lane with one ballot, builds the lane's state from the segment's base
// (base[row] + sum of change[row][n] count_n, a dense product: rows and counts need no
// lists and no read-modify-write chains), and takes the rates, sums and choice of the
// thread method: about 150 instructions and 450 cycles for six transitions, against
// 2,800 cycles for a pass over transitions, counts and sums in shared memory one by
// one.  Where every change is -1, 0 or 1 and at most 16 rows move, the state comes from
// byte sums instead: a lane's choice as one byte (change + 1) a row, four rows a word,
// summed over the lanes below in log2(SEG) shuffles a word (at most 64 a byte).  EXACT (SEG = 32): the clock of each lane's draw in binary64 (tau of its state,
// summed exactly in Q62; a decision is certain outside (k + 2) 2^-52), for node-days
// whose binary32 clock was too close to call.  Otherwise tau~ = E~ / a0~ (neglog_f32:
// 16u) goes through a binary32 scan of the round, whose start is a binary32 pair:
// within (nt + 38)u t of the binary64 chain; it is taken in every pass, and the round
// ends once no choice before the first draw that is not a certain continue changes
// (rounds that rarely hold the day's end, a0 > 2 SEG, settle every choice first).
// Every lane returns its segment's transitions fired, or -1 (a clock decision too close
// to call, or a state out of bounds): base then no longer holds the day's start.
template <int L, int SEG, bool EXACT>
__device__ __forceinline__ int32_t gen_draws_node_day(const GenSsaArgs& a, const GenModelDev& m, const GenRepParams& p,
                                                      const float* S, const uint32_t* pk, const float (&kyf)[L],
                                                      float* xf, float* base, const double* y, uint32_t v, uint32_t rep, uint32_t k0,
                                                      uint32_t k1, bool live, float margin) {
  const unsigned full = 0xffffffffu;
  const unsigned seg = SEG == 32 ? full : ((1u << (SEG & 31)) - 1u);
  const int lane = threadIdx.x & 31, sl = lane & (SEG - 1), sb = lane & ~(SEG - 1);
  const unsigned below = ((1u << sl) - 1u) << sb;
  const int nt = a.nt, rows = a.dyn_rows;
  bool done = !live || nt == 0;
  int32_t result = 0, fired = 0;
  float hi = 2.0f, lo = 0.0f;
  uint64_t tq = 0;
  for (int r = rows; r < a.xrows; ++r) xf[r * kGenThreads] = base[r];   // rows no firing changes
  for (uint32_t kb = 0; !__all_sync(full, done); kb += SEG) {
    if (!done && kb >= kGenSpecMaxSteps) { done = true; result = -1; }
    const uint4 w = philox10(make_uint4(v, (uint32_t)a.day, kb + (uint32_t)sl, rep), k0, k1);
    const uint64_t j52 = (((uint64_t)w.y << 32) | w.x) >> 12;
    const float Ef = EXACT ? 0.0f : neglog_f32(j52);
    const float u2f = f32_of_q53(((((((uint64_t)w.w) << 32) | w.z) >> 12) << 1) | 1ull);
    int choice = -2, e = SEG;
    float sc = 0.0f;
    bool bad = false, valid = false, sure = false;
    for (int it = 0; it <= SEG; ++it) {
      float least = 0.0f, most = 0.0f;
      if (a.pk_words > 0) {
        const float back = __int2float_rn(sl);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          if (q >= a.pk_words) break;
          const uint32_t own = choice >= 0 ? pk[choice * a.pk_words + q] : 0x01010101u;
          uint32_t sum = own;
#pragma unroll
          for (int o = 1; o < SEG; o <<= 1) {
            const uint32_t t = __shfl_up_sync(full, sum, o, SEG);
            if (sl >= o) sum += t;
          }
          sum -= own;
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const int r = 4 * q + i;
            if (r < rows) {
              const float x = __fadd_rn(base[r], __fsub_rn(__uint2float_rn((sum >> (8 * i)) & 0xffu), back));
              least = fminf(least, x);
              most = fmaxf(most, x);
              xf[r * kGenThreads] = x;
            }
          }
        }
      } else {
        float cnt[L];
#pragma unroll
        for (int n = 0; n < L; ++n)
          cnt[n] = n < nt ? __int2float_rn(__popc(__ballot_sync(full, choice == n) & below)) : 0.0f;
        for (int r = 0; r < rows; ++r) {
          float x = base[r];
          const float* Sr = S + r * L;
#pragma unroll
          for (int n = 0; n < L; ++n) x = __fmaf_rn(Sr[n], cnt[n], x);
          least = fminf(least, x);
          most = fmaxf(most, x);
          xf[r * kGenThreads] = x;
        }
      }
      bad = least < 0.0f || most >= kGenBigCount;
      float P[L];
      const float a0 = gen_sums_f32<L>(a, kyf, xf, P);
      valid = !done && !bad && a0 > 0.0f;
      int next = -1;
      if (valid) {
        next = gen_select_f32<L>(nt, P, __fmul_rn(a0, u2f));
        // (a draw that cannot be a certain continue ends the day: its choice is not needed)
        if (next < 0 && (EXACT || a0 >= kGenSmallA0)) {
          column_to_int(xf, m.nc);
          next = gen_exact_choice(m, p, reinterpret_cast<const int32_t*>(xf), kGenThreads, y, uniform_open(w.z, w.w));
          column_to_float(xf, m.nc);
        }
      }
      const bool changed = next != choice;
      if ((EXACT || __any_sync(full, valid && a0 > 2.0f * SEG)) && it < SEG && __any_sync(full, changed)) {
        choice = next;
        continue;
      }
      if (EXACT) { choice = next; break; }
      sc = valid ? fminf(__fmul_rn(Ef, rcp_approx(a0)), 4.0f) : 0.0f;
#pragma unroll
      for (int o = 1; o < SEG; o <<= 1) {
        const float t = __shfl_up_sync(full, sc, o, SEG);
        if (sl >= o) sc = __fadd_rn(sc, t);
      }
      const float d = __fadd_rn(__fadd_rn(__fsub_rn(hi, 3.0f), lo), sc);
      const bool cont = valid && a0 >= kGenSmallA0 && d <= -margin;
      sure = !bad && (!valid || d >= margin);
      const unsigned notcont = (__ballot_sync(full, !cont) >> sb) & seg;
      e = notcont ? __ffs(notcont) - 1 : SEG;
      const unsigned diff = (__ballot_sync(full, changed) >> sb) & seg & (e < SEG ? ((1u << e) - 1u) : seg);
      choice = next;
      if (__all_sync(full, done || diff == 0u)) break;
    }
    if (EXACT) {
      // tau of the lane's draw in binary64, the round's clock exactly in Q62
      uint64_t q = 0;
      if (valid) {
        column_to_int(xf, m.nc);
        double A = 0.0;
        for (int j = 0; j < nt; ++j) {
          const double aj = gen_rate(m, p, reinterpret_cast<const int32_t*>(xf), kGenThreads, y, j);
          A = j == 0 ? aj : __dadd_rn(A, aj);
        }
        column_to_float(xf, m.nc);
        const double tau = div_pos(neglog_u(j52), A);
        q = q62_of_f64(le_nonneg(tau, 1.5) ? tau : 1.5);
      }
#pragma unroll
      for (int o = 1; o < SEG; o <<= 1) {
        const uint64_t t = __shfl_up_sync(full, q, o, SEG);
        if (sl >= o) q += t;
      }
      const uint64_t t = tq + q, close = ((uint64_t)kb + (uint64_t)sl + 2ull) << 10;   // (k + 2) 2^-52
      sure = !bad && (!valid || t >= kQ62One + close);
      const unsigned notcont = __ballot_sync(full, !(valid && t + close < kQ62One));
      e = notcont ? __ffs(notcont) - 1 : SEG;
      tq = __shfl_sync(full, t, SEG - 1);
    }
    // the round's outcome per segment: the state before draw e, or after the last one
    const unsigned sures = (__ballot_sync(full, sure) >> sb) & seg;
    const int src = sb + (e < SEG ? e : SEG - 1);
    const int last = __shfl_sync(full, choice, src);
    const float round = __shfl_sync(full, sc, src);
    __syncwarp();
    if (!done) {
      for (int r = sl; r < rows; r += SEG) {
        float x = xf[r * kGenThreads + (src - lane)];
        if (e == SEG && last >= 0) x = __fadd_rn(x, S[r * L + last]);   // every lane fired
        base[r] = x;
      }
      if (e < SEG) {
        result = ((sures >> e) & 1u) ? fired + e : -1;
        done = true;
      } else {
        const float hn = __fadd_rn(hi, round);
        lo = __fadd_rn(lo, __fsub_rn(round, __fsub_rn(hn, hi)));
        hi = hn;
        fired += SEG;
      }
    }
    __syncwarp();
  }
  return result;
}

// Bound by the latency of the longest chain of a launch (about 10 us of it fixed: the
// model's copy, order, counts, variables and constants in sequence).  Measured per run,
// one GB300, against the kernel this replaced (transitions walked in shared memory, one
// block of 128 nodes each): SIR 2,000 nodes x 60 days 2.0 -> 1.2 ms, Erlang 1,500 x 40
// 13.8 -> 3.3 ms, SEIRS midpoint 37,000 x 365 26.1 -> 16.4 ms, SISe3 37,000 x 365
// 20.1 -> 13.5 ms; with the byte sums, overlapped starts and a kept graph since then
// 0.91, 2.8, 14.0 and 11.0-13.4 ms (SIR 0.77 and SEIRS 13.0 with k_gen_events_small).
//
// The stochastic step: warps of a resident grid (as node_day_dealt deals its units) take
// the warp nodes first (largest first, a node's replicates together), then units of four
// nodes for the segment method, then units of 32 for the thread method.
template <int L>
__global__ void __launch_bounds__(kGenThreads, 4) k_gen_ssa(GenSsaArgs a) {
  extern __shared__ int4 smem4[];
  GenModelDev& m = *reinterpret_cast<GenModelDev*>(smem4);
  char* sp = reinterpret_cast<char*>(smem4) + sizeof(GenModelDev);
  grid_dependents_launch();
  copy16(&m, a.model, (int)(sizeof(GenModelDev) / 16));
  // the change tables: [dyn_rows][L], the thread method's [nt], bytes [nt][pk_words], longer lists
  float* S = reinterpret_cast<float*>(sp);
  int4* chg = reinterpret_cast<int4*>(S + a.dyn_rows * L);
  const uint32_t* pk = reinterpret_cast<const uint32_t*>(chg + a.nt);
  const int2* more = reinterpret_cast<const int2*>(pk + a.nt * a.pk_words + (a.nt * a.pk_words & 1));
  copy16(S, a.tab, a.tab16);
  sp += (size_t)a.tab16 * 16;
  double* ctau = reinterpret_cast<double*>(sp);                 // [threads]: per lane
  sp += kGenThreads * sizeof(double);
  double* rates = reinterpret_cast<double*>(sp);                // [nt][threads], then partial sums
  sp += (size_t)2 * a.nt * kGenThreads * sizeof(double);
  int32_t* rows = reinterpret_cast<int32_t*>(sp);               // [threads / kGenSeg][kGenMaxComp]: day-start counts
  sp += (kGenThreads / kGenSeg) * kGenMaxComp * sizeof(int32_t);
  int32_t* cch = reinterpret_cast<int32_t*>(sp);                // [threads]: per lane
  sp += kGenThreads * sizeof(int32_t);
  float* kys = reinterpret_cast<float*>(sp);                    // [threads / kGenSeg][L]: a segment's constants
  sp += (kGenThreads / kGenSeg) * L * sizeof(float);
  float* bases = reinterpret_cast<float*>(sp);                  // [threads / kGenSeg][xrows]
  sp += (size_t)(kGenThreads / kGenSeg) * a.xrows * sizeof(float);
  float* xfs = reinterpret_cast<float*>(sp);                    // [xrows][threads]
  sp += (size_t)a.xrows * kGenThreads * sizeof(float);
  int32_t* xs = reinterpret_cast<int32_t*>(sp);                 // [nc][threads]
  __syncthreads();
  const unsigned full = 0xffffffffu;
  const int nc = m.nc, nt = a.nt, ny = m.ny, N = a.N;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  // 32-bit unit numbers: gen_create bounds R nc N by 2^31
  constexpr int kPer = 32 / kGenSeg;
  const uint32_t T = gridDim.x * kGenWarps, R = (uint32_t)a.R;
  const uint32_t uw = R * (uint32_t)a.n_big, ug = R * (((uint32_t)a.n_mid + kPer - 1) / kPer);
  const uint32_t units = uw + ug + R * (((uint32_t)(N - a.n_big - a.n_mid) + 31) / 32);
  const uint32_t k0 = (uint32_t)a.seed, k1 = (uint32_t)(a.seed >> 32), day = (uint32_t)a.day;
  const RateRow RR{rates + threadIdx.x, rates + (size_t)nt * kGenThreads + threadIdx.x, kGenThreads};
  const bool midpoint = m.y_source == kGenYMidpoint, pre_event = m.y_source == kGenYPreEvent;
  float* xf = xfs + threadIdx.x;
  int32_t* xi = reinterpret_cast<int32_t*>(xf);
  grid_dependency_wait();                                       // counts and variables of the previous step
  for (uint32_t u = (uint32_t)warp * gridDim.x + blockIdx.x; u < units; u += T) {
    // role 0: a warp node; 1: four nodes on segments; 2: 32 nodes
    const int role = u < uw ? 0 : (u < uw + ug ? 1 : 2);
    const uint32_t ut = role == 0 ? u : (role == 1 ? u - uw : u - uw - ug);
    const uint32_t gi = R == 1 ? ut : ut / R;
    const int r = (int)(ut - gi * R);
    const int i = role == 0 ? (int)gi
                            : (role == 1 ? a.n_big + (int)gi * kPer + lane / kGenSeg
                                         : a.n_big + a.n_mid + (int)gi * 32 + lane);
    const bool has = role == 0 || i < (role == 1 ? a.n_big + a.n_mid : N);
    const int v = has ? a.order[i] : 0;
    const GenRepParams& p = a.params[r];
    const uint32_t rep = (uint32_t)(a.rep_base + r);
    int32_t* X = a.counts + (size_t)r * nc * N + v;
    double* Y = a.y + (size_t)r * ny * N + v;
    // lanes per node, the lane's index among them and the node's first lane
    const int width = role == 0 ? 32 : (role == 1 ? kGenSeg : 1);
    const int sl = lane & (width - 1), sb = lane & ~(width - 1);
    const int slot = warp * kPer + (role == 1 ? lane / kGenSeg : 0);
    int32_t* row = rows + slot * kGenMaxComp;                   // roles 0 and 1: the node's counts
    if (has)
      for (int c = sl; c < nc; c += width) {
        const int32_t x = __ldcg(X + (size_t)c * N);
        if (role == 2) xi[c * kGenThreads] = x; else row[c] = x;
      }
    __syncwarp();
    const int32_t* x0 = role == 2 ? xi : row;
    const int xst = role == 2 ? kGenThreads : 1;
    // continuous variables, shared out over the node's lanes: day - 1's update from its
    // post-event counts, or the midpoint with the sums saved at its start; then frozen
    double y[kGenMaxCont];
    for (int q = 0; q < ny; ++q) {
      double yq = 0.0;
      if (has && (q & (width - 1)) == sl) {
        yq = __ldcg(Y + (size_t)q * N);
        double* M = a.mid + ((size_t)r * ny + q) * 2 * N + v;
        double U = 0.0, D = 0.0;
        if (a.prologue || midpoint) {
          U = u2d_exact(mask_sum(x0, xst, m.num[q], nc));
          D = u2d_exact(mask_sum(x0, xst, m.den[q], nc));
        }
        if (a.prologue) {
          yq = gen_y_next(m, p, q, a.day - 1, yq, midpoint ? __dmul_rn(0.5, __dadd_rn(__ldcg(M), U)) : U,
                          midpoint ? __dmul_rn(0.5, __dadd_rn(__ldcg(M + N), D)) : D);
          Y[(size_t)q * N] = yq;
        }
        if (midpoint) { M[0] = U; M[N] = D; }
      }
      y[q] = role == 2 ? yq : __shfl_sync(full, yq, sb + (q & (width - 1)));
    }
    // binary32 constants, populations and counts (roles 0 and 1: the segment's base)
    bool ok = true;
    float kyf[L];
    if (role == 2) {
#pragma unroll
      for (int j = 0; j < L; ++j) {
        kyf[j] = 0.0f;
        if (j < nt) ok = gen_const_f32(p.rate[j], a.fy[j] >= 0, a.fy[j] >= 0 ? y[a.fy[j]] : 0.0, kyf[j]) && ok;
      }
    } else {
      for (int j = sl; j < nt; j += width) {
        float c;
        ok = gen_const_f32(p.rate[j], m.fy[j] >= 0, m.fy[j] >= 0 ? y[m.fy[j]] : 0.0, c) && ok;
        kys[slot * L + j] = c;
      }
      __syncwarp();
#pragma unroll
      for (int j = 0; j < L; ++j) kyf[j] = j < nt ? kys[slot * L + j] : 0.0f;
    }
    float* base = bases + slot * a.xrows;
    long long tot = 0;
    if (has)
      for (int c = 0; c < nc; ++c) tot += x0[c * xst];
    ok = ok && tot < (1 << 21);
    if (has && ok) {
      for (int q = sl; q < a.npop; q += width) {
        const float P = __int2float_rn((int32_t)mask_sum(x0, xst, a.pops[q], nc));
        if (role == 2) xf[(nc + q) * kGenThreads] = P; else base[nc + q] = P;
      }
      if (role == 2) {
        column_to_float(xf, nc);
        xf[(nc + a.npop) * kGenThreads] = 1.0f;
        xf[(nc + a.npop + 1) * kGenThreads] = 0.0f;
      } else {
        for (int c = sl; c < nc; c += width) base[c] = __int2float_rn(row[c]);
        if (sl == 0) { base[nc + a.npop] = 1.0f; base[nc + a.npop + 1] = 0.0f; }
      }
    }
    __syncwarp();
    int32_t f = has ? -1 : 0;
    if (role == 2) {
      if (has && ok)
        f = nt == 0 ? 0 : gen_thread_node_day<L>(a, m, p, chg, more, kyf, xf, y, (uint32_t)v, rep, k0, k1, a.margin_f);
      if (has && f >= 0) {
        column_to_int(xf, nc);
        for (int c = 0; c < nc; ++c) X[(size_t)c * N] = xi[c * kGenThreads];
      }
    } else if (role == 1) {
      const unsigned oks = __ballot_sync(full, ok);
      const bool live = has && ((oks >> sb) & ((1u << kGenSeg) - 1u)) == (1u << kGenSeg) - 1u;
      const int32_t g = gen_draws_node_day<L, kGenSeg, false>(a, m, p, S, pk, kyf, xf, base, y, (uint32_t)v, rep, k0, k1,
                                                              live, a.margin_f);
      if (live) f = g;
    } else if (__all_sync(full, ok)) {
      f = gen_draws_node_day<L, 32, false>(a, m, p, S, pk, kyf, xf, base, y, (uint32_t)v, rep, k0, k1, true, a.margin_f);
    }
    if (role != 2 && has && f >= 0)
      for (int c = sl; c < nc; c += width) {
        const int32_t x = (int32_t)base[c];
        row[c] = x;
        X[(size_t)c * N] = x;
      }
    __syncwarp();
    if (pre_event && has && f >= 0)
      for (int q = sl; q < ny; q += width)
        Y[(size_t)q * N] = gen_y_next(m, p, q, a.day, y[q], u2d_exact(mask_sum(x0, xst, m.num[q], nc)),
                                      u2d_exact(mask_sum(x0, xst, m.den[q], nc)));
    // node-days handed back: the whole warp runs each in turn from the day's start (its
    // global counts), with the binary64 clock, then with the binary64 method
    unsigned need = __ballot_sync(full, has && f < 0 && sl == 0);
    while (need) {
      const int l = __ffs(need) - 1;
      need &= need - 1;
      const int vl = __shfl_sync(full, v, l);
      double yl[kGenMaxCont];
      for (int q = 0; q < ny; ++q) yl[q] = __shfl_sync(full, y[q], l);
      float kl[L];
#pragma unroll
      for (int j = 0; j < L; ++j) kl[j] = __shfl_sync(full, kyf[j], l);
      const bool okl = __shfl_sync(full, role == 2 ? ok : tot < (1 << 21), l) &&
                       (role == 2 || !__any_sync(full, !ok && sb == l));
      int32_t* Xl = a.counts + (size_t)r * nc * N + vl;
      int32_t* rl = rows + warp * kPer * kGenMaxComp;           // the warp's first slot: its own node is stored, or this one
      float* bl = bases + warp * kPer * a.xrows;
      __syncwarp();
      if (lane < nc) rl[lane] = __ldcg(Xl + (size_t)lane * N);
      __syncwarp();
      int32_t n = -1;
      if (okl) {
        for (int q = lane; q < a.npop; q += 32) bl[nc + q] = __int2float_rn((int32_t)mask_sum(rl, 1, a.pops[q], nc));
        if (lane < nc) bl[lane] = __int2float_rn(rl[lane]);
        if (lane == 0) { bl[nc + a.npop] = 1.0f; bl[nc + a.npop + 1] = 0.0f; }
        __syncwarp();
        n = gen_draws_node_day<L, 32, true>(a, m, p, S, pk, kl, xf, bl, yl, (uint32_t)vl, rep, k0, k1, true, 0.0f);
        if (n >= 0 && lane < nc) rl[lane] = (int32_t)bl[lane];
        __syncwarp();
      }
      if (n < 0)
        n = (int32_t)gen_seg_node_day<32>(m, p, xs + threadIdx.x, rl, kGenThreads, RR, ctau + warp * 32,
                                          cch + warp * 32, yl, (uint32_t)vl, day, rep, k0, k1, lane, 0, true);
      if (lane < nc) Xl[(size_t)lane * N] = rl[lane];
      if (pre_event && lane < ny) {
        double* Yl = a.y + ((size_t)r * ny + lane) * N + vl;
        *Yl = gen_y_next(m, p, lane, a.day, *Yl, u2d_exact(mask_sum(rl, 1, m.num[lane], nc)),
                         u2d_exact(mask_sum(rl, 1, m.den[lane], nc)));
      }
      if (sb == l) f = n;
      __syncwarp();
    }
    const uint32_t tot_fired = __reduce_add_sync(full, has && sl == 0 ? (uint32_t)f : 0u);
    if (lane == 0 && tot_fired) atomicAdd(a.ctr + (size_t)r * 4, (unsigned long long)tot_fired);
    __syncwarp();                                               // rows, bases and columns are reused by the next unit
  }
}

// The binary64 methods only (GEN_OPT_CLOCK_MARGIN 0): warp and group nodes by the
// segment method, the rest one per thread.
__global__ void __maxnreg__(128) k_gen_ssa_exact(GenSsaArgs a) {
  extern __shared__ int4 smem4[];
  GenModelDev& m = *reinterpret_cast<GenModelDev*>(smem4);
  char* sp = reinterpret_cast<char*>(smem4) + sizeof(GenModelDev);
  grid_dependents_launch();
  grid_dependency_wait();
  GenRepParams& p = *reinterpret_cast<GenRepParams*>(sp);
  sp += sizeof(GenRepParams);
  double* ctau = reinterpret_cast<double*>(sp);                 // [threads]: per lane
  sp += kGenThreads * sizeof(double);
  const int r = blockIdx.y;
  copy16(&m, a.model, (int)(sizeof(GenModelDev) / 16));
  copy16(&p, a.params + r, (int)(sizeof(GenRepParams) / 16));
  __syncthreads();
  const int nc = m.nc, nt = m.nt, ny = m.ny, N = a.N;
  double* rates = reinterpret_cast<double*>(sp);                // [nt][threads], then partial sums
  sp += (size_t)2 * nt * kGenThreads * sizeof(double);
  int32_t* sbase = reinterpret_cast<int32_t*>(sp);              // [warps][4 segments][kGenMaxComp]
  sp += kGenWarps * (32 / kGenSeg) * kGenMaxComp * sizeof(int32_t);
  int32_t* cch = reinterpret_cast<int32_t*>(sp);                // [threads]: per lane
  sp += kGenThreads * sizeof(int32_t);
  int32_t* xs = reinterpret_cast<int32_t*>(sp);                 // [nc][threads]
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int stride = blockDim.x;
  const int b = (int)blockIdx.x;
  // units: warp nodes (one per warp), group nodes (four per warp), thread nodes
  const int kind = b < a.warp_blocks ? 0 : (b < a.warp_blocks + a.group_blocks ? 1 : 2);
  const int sl = kind == 0 ? lane : (kind == 1 ? (lane & (kGenSeg - 1)) : 0);
  const int sb = kind == 1 ? (lane & ~(kGenSeg - 1)) : 0;
  int v = -1;
  if (kind == 0) {
    const int u = b * kGenWarps + warp;
    if (u < a.n_big) v = a.order[u];
  } else if (kind == 1) {
    const int g = ((b - a.warp_blocks) * kGenWarps + warp) * (32 / kGenSeg) + (lane / kGenSeg);
    if (g < a.n_mid) v = a.order[a.n_big + g];
  } else {
    const int i = a.n_big + a.n_mid + (b - a.warp_blocks - a.group_blocks) * kGenThreads + (int)threadIdx.x;
    if (i < N) v = a.order[i];
  }
  const bool coop = kind != 2;
  // a cooperative warp runs when any of its segments has a node; a thread when it has one
  const bool run = coop ? __any_sync(0xffffffffu, v >= 0) : v >= 0;
  uint32_t fired = 0;
  if (run) {
    const bool has = v >= 0;
    int32_t* x = xs + threadIdx.x;
    int32_t* base = sbase + (warp * (32 / kGenSeg) + (kind == 1 ? lane / kGenSeg : 0)) * kGenMaxComp;
    const RateRow R{rates + threadIdx.x, rates + (size_t)nt * kGenThreads + threadIdx.x, kGenThreads};
    int32_t* X = a.counts + (size_t)r * nc * N;
    if (coop) {
      if (has)
        for (int c = sl; c < nc; c += (kind == 0 ? 32 : kGenSeg)) base[c] = X[(size_t)c * N + v];
      __syncwarp();
    } else {
      for (int c = 0; c < nc; ++c) x[c * stride] = X[(size_t)c * N + v];
    }
    // the node's counts at the start of the day, as this lane sees them
    const int32_t* x0 = coop ? base : x;
    const int s0 = coop ? 1 : stride;
    double y[kGenMaxCont];
    double* Y = a.y + (size_t)r * ny * N;
    const bool writer = has && (!coop || sl == 0);
    if (has) {
      for (int q = 0; q < ny; ++q) y[q] = Y[(size_t)q * N + v];
      if (a.prologue) {
        // day - 1's continuous update from its post-event counts (and, for the
        // midpoint, the sums saved at its start), then frozen for this day
        for (int q = 0; q < ny; ++q) {
          double U = u2d_exact(mask_sum(x0, s0, m.num[q], nc));
          double D = u2d_exact(mask_sum(x0, s0, m.den[q], nc));
          if (m.y_source == kGenYMidpoint) {
            const double* M = a.mid + ((size_t)r * ny + q) * 2 * N;
            U = __dmul_rn(0.5, __dadd_rn(M[v], U));
            D = __dmul_rn(0.5, __dadd_rn(M[(size_t)N + v], D));
          }
          y[q] = gen_y_next(m, p, q, a.day - 1, y[q], U, D);
        }
      }
    }
    if (coop) __syncwarp();
    if (writer) {
      if (a.prologue)
        for (int q = 0; q < ny; ++q) Y[(size_t)q * N + v] = y[q];
      if (m.y_source == kGenYMidpoint)
        for (int q = 0; q < ny; ++q) {
          double* M = a.mid + ((size_t)r * ny + q) * 2 * N;
          M[v] = u2d_exact(mask_sum(x0, s0, m.num[q], nc));
          M[(size_t)N + v] = u2d_exact(mask_sum(x0, s0, m.den[q], nc));
        }
    }
    const uint32_t rep = (uint32_t)(a.rep_base + r), k0 = (uint32_t)a.seed, k1 = (uint32_t)(a.seed >> 32);
    const uint32_t vv = (uint32_t)(has ? v : 0);
    if (kind == 0)
      fired = gen_seg_node_day<32>(m, p, x, base, stride, R, ctau + warp * 32, cch + warp * 32, y, vv, (uint32_t)a.day,
                                   rep, k0, k1, sl, sb, has);
    else if (kind == 1)
      fired = gen_seg_node_day<kGenSeg>(m, p, x, base, stride, R, ctau + warp * 32 + sb, cch + warp * 32 + sb, y, vv,
                                        (uint32_t)a.day, rep, k0, k1, sl, sb, has);
    else
      fired = gen_node_day(m, p, x, stride, R, y, (uint32_t)v, (uint32_t)a.day, rep, k0, k1);
    if (writer) {
      for (int c = 0; c < nc; ++c) X[(size_t)c * N + v] = x0[c * s0];
      if (m.y_source == kGenYPreEvent) {
        for (int q = 0; q < ny; ++q) {
          const double U = u2d_exact(mask_sum(x0, s0, m.num[q], nc));
          const double D = u2d_exact(mask_sum(x0, s0, m.den[q], nc));
          Y[(size_t)q * N + v] = gen_y_next(m, p, q, a.day, y[q], U, D);
        }
      }
    }
    if (coop && !writer) fired = 0;
  }
  const uint32_t tot = __reduce_add_sync(0xffffffffu, fired);
  if (lane == 0 && tot) atomicAdd(a.ctr + (size_t)r * 4, (unsigned long long)tot);
}

// `take` of the animals counted by h (their sum, avail, above `take`), uniformly and one
// at a time, from the event's word stream, whose first Philox block comes with the call
// (w).  A draw is compared with the running sums of what is left, all at once; WIDE, for
// a sum past 32 bits (entries alone can get there), walks the compartments instead.
template <bool WIDE, int C>
__device__ __forceinline__ void gen_take(const int32_t (&h)[C], int64_t avail, int take, uint4 w, uint32_t e,
                                         uint32_t tag, uint32_t rep, uint32_t k0, uint32_t k1, int32_t (&took)[C]) {
  uint32_t cum[C];
#pragma unroll
  for (int c = 0; c < C; ++c) {
    cum[c] = (uint32_t)h[c] + (c && !WIDE ? cum[c > 0 ? c - 1 : 0] : 0u);
  }
  uint32_t wq = 0;
  auto next = [&]() -> uint32_t {
    const uint32_t s = wq & 3u;
    if (s == 0u && wq) w = philox10(make_uint4(e, tag, wq >> 2, rep), k0, k1);
    ++wq;
    return s == 0 ? w.x : s == 1 ? w.y : s == 2 ? w.z : w.w;
  };
#pragma unroll 1
  for (int t = 0; t < take; ++t) {
    uint32_t slot = lemire((uint32_t)(avail - t), next);
    bool open = true;
#pragma unroll
    for (int c = 0; c < C; ++c) {
      const bool hit = open && slot < cum[c];
      if (WIDE) {
        open = open && !hit;
        slot -= open ? cum[c] : 0u;
      }
      cum[c] -= hit ? 1u : 0u;
    }
  }
#pragma unroll
  for (int c = 0; c < C; ++c) took[c] = h[c] - (int32_t)(cum[c] - (c && !WIDE ? cum[c > 0 ? c - 1 : 0] : 0u));
}

// One thread per component of the day's transfer graph: its events in input
// order (no other thread touches its nodes this day).  Components (largest first)
// are dealt lane-major over the grid's warps: component i runs on lane i / W of
// warp i mod W (W warps in all), so the largest W each have a warp to themselves
// and no warp serialises several long divergent chains.  The counts of the node an
// event samples from stay in a shared-memory row across consecutive events at
// that node; transfers add to the destination in global memory (a destination is
// never the node in the row, and the row is written back before another node is
// loaded).
__global__ void __launch_bounds__(kGenThreads) k_gen_events(GenEvArgs a) {
  __shared__ GenModelDev m;
  __shared__ int32_t cache[kGenMaxComp * kGenThreads];
  grid_dependents_launch();
  copy16(&m, a.model, (int)(sizeof(GenModelDev) / 16));
  __syncthreads();
  const int r = blockIdx.y, nc = m.nc, N = a.N;
  const int W = (int)gridDim.x * (int)(blockDim.x >> 5);
  const int ci = (int)(threadIdx.x & 31) * W + (int)blockIdx.x * (int)(blockDim.x >> 5) + (int)(threadIdx.x >> 5);
  int32_t* cc = cache + threadIdx.x;
  const int S = kGenThreads;
  uint32_t applied = 0, clamped = 0, skipped = 0;
  if (ci < a.ncomp) {
    int32_t* X = a.counts + (size_t)r * nc * N;
    const uint32_t rep = (uint32_t)(a.rep_base + r), k0 = (uint32_t)a.seed, k1 = (uint32_t)(a.seed >> 32);
    int cur = -1;
    const int p1 = a.comp_off[a.comp0 + ci + 1];
    int pi = a.comp_off[a.comp0 + ci];
    int e_next = 0;
    int4 rec_next = make_int4(0, 0, 0, 0);
    if (pi < p1) { e_next = __ldg(a.comp_ev + pi); rec_next = __ldg(a.rec + pi); }
    grid_dependency_wait();                          // the stochastic step's counts
    for (; pi < p1; ++pi) {
      const int e = e_next;
      const int4 rec = rec_next;
      if (pi + 1 < p1) { e_next = __ldg(a.comp_ev + pi + 1); rec_next = __ldg(a.rec + pi + 1); }
      const int node = rec.x, dest = rec.y, n = rec.z;
      const int kind = rec.w & 0xff, sel = (rec.w >> 8) & 0xff, sh = (rec.w >> 16) & 0xff;
      const uint32_t mask = m.select[sel];
      const int8_t* off = m.shift[sh];
      if (node != cur) {
        if (cur >= 0)
          for (int c = 0; c < nc; ++c) X[(size_t)c * N + cur] = cc[c * S];
        for (int c = 0; c < nc; ++c) cc[c * S] = X[(size_t)c * N + node];
        cur = node;
      }
      if (kind == SIM_ENTER) {
        const int c0 = __ffs(mask) - 1;
        cc[(c0 + off[c0]) * S] += n;
        ++applied;
        continue;
      }
      long long avail = 0;
      for (int c = 0; c < nc; ++c)
        if (mask >> c & 1u) avail += cc[c * S];
      int take = n;
      if ((long long)n > avail) {
        if (a.underflow_error) {
          ++skipped;
          atomicOr(a.err, 1);
          continue;
        }
        take = (int)avail;
        ++clamped;
      }
      uint4 buf = make_uint4(0, 0, 0, 0);
      uint32_t wq = 0;
      auto next = [&]() -> uint32_t {
        if ((wq & 3u) == 0u) buf = philox10(make_uint4((uint32_t)e, (uint32_t)a.day | kEventTag, wq >> 2, rep), k0, k1);
        const uint32_t s = wq & 3u;
        ++wq;
        return s == 0 ? buf.x : s == 1 ? buf.y : s == 2 ? buf.z : buf.w;
      };
      for (int t = 0; t < take; ++t) {
        uint32_t slot = lemire((uint32_t)(avail - t), next);
        int got = 0;
        for (int c = 0; c < nc; ++c) {
          if (!(mask >> c & 1u)) continue;
          const uint32_t have = (uint32_t)cc[c * S];
          if (slot < have) { got = c; break; }
          slot -= have;
        }
        cc[got * S] -= 1;
        if (kind == SIM_INTERNAL) cc[(got + off[got]) * S] += 1;
        else if (kind == SIM_EXTERNAL) X[(size_t)(got + off[got]) * N + dest] += 1;
      }
      ++applied;
    }
    if (cur >= 0)
      for (int c = 0; c < nc; ++c) X[(size_t)c * N + cur] = cc[c * S];
  }
  grid_dependency_wait();                            // threads without a component too
  const uint32_t sa = __reduce_add_sync(0xffffffffu, applied);
  const uint32_t sc = __reduce_add_sync(0xffffffffu, clamped);
  const uint32_t ss = __reduce_add_sync(0xffffffffu, skipped);
  if ((threadIdx.x & 31) == 0) {
    unsigned long long* C = a.ctr + (size_t)r * 4;
    if (sa) atomicAdd(C + 1, (unsigned long long)sa);
    if (sc) atomicAdd(C + 2, (unsigned long long)sc);
    if (ss) atomicAdd(C + 3, (unsigned long long)ss);
  }
}

// The event step for models of up to four compartments, dealt as in k_gen_events.  What
// bounds it is one thread's chain of latencies, so nothing in it waits that need not:
// the records come two events ahead, the next event's first Philox block and the counts
// of the node it samples one ahead (the first of them before the stochastic step is
// done); the counts of the node being sampled stay in registers with the running sums
// that a draw is compared with all at once; transfers leave as reductions, which nobody
// waits for.  A destination is never the node in the registers, and a node that the
// current event adds to is not read ahead.  A launch of a SEIRS day (about 2,600
// components): 9.6 -> 8.4 us; a year of it 13.9 -> 12.7 ms, 60 days of SIR with 2,000
// nodes 0.92 -> 0.77 ms.  For more compartments the fixed work per event outgrows what
// the row in shared memory costs on the long chains of a hub herd: six compartments,
// 37,000 herds, a year: 11.2 -> 10.7 ms on some schedules, 13.4 -> 13.9 on those with
// longer chains, so those keep k_gen_events.
template <int C>
__global__ void __launch_bounds__(kGenThreads) k_gen_events_small(GenEvArgs a) {
  __shared__ GenModelDev m;
  grid_dependents_launch();
  copy16(&m, a.model, (int)(sizeof(GenModelDev) / 16));
  __syncthreads();
  const int r = blockIdx.y, nc = m.nc, N = a.N;
  const int W = (int)gridDim.x * (int)(blockDim.x >> 5);
  const int ci = (int)(threadIdx.x & 31) * W + (int)blockIdx.x * (int)(blockDim.x >> 5) + (int)(threadIdx.x >> 5);
  uint32_t applied = 0, clamped = 0, skipped = 0;
  if (ci < a.ncomp) {
    int32_t* X = a.counts + (size_t)r * nc * N;
    const uint32_t rep = (uint32_t)(a.rep_base + r);
    uint32_t k0 = (uint32_t)a.seed, k1 = (uint32_t)(a.seed >> 32);
    const uint32_t tag = (uint32_t)a.day | kEventTag;
    auto load_row = [&](int v, int32_t (&x)[C]) {
#pragma unroll
      for (int c = 0; c < C; ++c) x[c] = c < nc ? __ldcg(X + (size_t)c * N + v) : 0;
    };
    auto store_row = [&](int v, const int32_t (&x)[C]) {
#pragma unroll
      for (int c = 0; c < C; ++c)
        if (c < nc) X[(size_t)c * N + v] = x[c];
    };
    int pi = a.comp_off[a.comp0 + ci];
    const int p1 = a.comp_off[a.comp0 + ci + 1];
    int4 rec = __ldg(a.rec + pi), rec1 = rec;        // a component has at least one event
    int e = __ldg(a.comp_ev + pi), e1 = e;
    if (pi + 1 < p1) { rec1 = __ldg(a.rec + pi + 1); e1 = __ldg(a.comp_ev + pi + 1); }
    uint4 w = philox10(make_uint4((uint32_t)e, tag, 0u, rep), k0, k1);
    grid_dependency_wait();                          // the stochastic step's counts
    int32_t x[C];
    load_row(rec.x, x);
#pragma unroll 1
    for (; pi < p1; ++pi) {
      asm volatile("" : "+r"(k0), "+r"(k1));        // keep the ten round keys out of registers
      int4 rec2 = rec1;
      int e2 = e1;
      if (pi + 2 < p1) { rec2 = __ldg(a.rec + pi + 2); e2 = __ldg(a.comp_ev + pi + 2); }
      const int node = rec.x, dest = rec.y, n = rec.z;
      const int kind = rec.w & 0xff, sel = (rec.w >> 8) & 0xff, sh = (rec.w >> 16) & 0xff;
      const bool move = pi + 1 < p1 && rec1.x != node;
      const bool ahead = move && !(kind == SIM_EXTERNAL && dest == rec1.x);
      int32_t nx[C];
      if (ahead) load_row(rec1.x, nx);
      const uint4 w1 = philox10(make_uint4((uint32_t)e1, tag, 0u, rep), k0, k1);
      const uint32_t mask = m.select[sel];
      const int8_t* off = m.shift[sh];
      if (kind == SIM_ENTER) {
        const int c0 = __ffs(mask) - 1, to = c0 + off[c0];
#pragma unroll
        for (int c = 0; c < C; ++c) x[c] += c == to ? n : 0;
        ++applied;
      } else {
        int32_t h[C], took[C];
        long long avail = 0;
        int kinds = 0;
#pragma unroll
        for (int c = 0; c < C; ++c) {
          h[c] = (mask >> c & 1u) ? x[c] : 0;
          avail += h[c];
          kinds += h[c] > 0 ? 1 : 0;
        }
        int take = n;
        bool apply = true;
        if ((long long)n > avail) {
          if (a.underflow_error) {
            ++skipped;
            atomicOr(a.err, 1);
            apply = false;
          } else {
            take = (int)avail;
            ++clamped;
          }
        }
        if (apply) {
          // every animal, or animals of one compartment: whatever the draws
          if (take == avail || kinds <= 1) {
#pragma unroll
            for (int c = 0; c < C; ++c) took[c] = h[c] > take ? take : h[c];
          } else if (avail >> 32) {
            gen_take<true, C>(h, avail, take, w, (uint32_t)e, tag, rep, k0, k1, took);
          } else {
            gen_take<false, C>(h, avail, take, w, (uint32_t)e, tag, rep, k0, k1, took);
          }
#pragma unroll
          for (int c = 0; c < C; ++c) x[c] -= took[c];
          if (kind != SIM_EXIT) {
#pragma unroll
            for (int c = 0; c < C; ++c) {
              if (!took[c]) continue;
              const int to = c + off[c];
              if (kind == SIM_EXTERNAL) {
                atomicAdd(&X[(size_t)to * N + dest], took[c]);
              } else {                               // never into the mask (checked at load)
#pragma unroll
                for (int k = 0; k < C; ++k) x[k] += k == to ? took[c] : 0;
              }
            }
          }
          ++applied;
        }
      }
      if (move) {
        store_row(node, x);
        if (!ahead) load_row(rec1.x, nx);
#pragma unroll
        for (int c = 0; c < C; ++c) x[c] = nx[c];
      } else if (pi + 1 >= p1) {
        store_row(node, x);
      }
      rec = rec1; e = e1; w = w1;
      rec1 = rec2; e1 = e2;
    }
  }
  grid_dependency_wait();                            // threads without a component too
  const uint32_t sa = __reduce_add_sync(0xffffffffu, applied);
  const uint32_t sc = __reduce_add_sync(0xffffffffu, clamped);
  const uint32_t ss = __reduce_add_sync(0xffffffffu, skipped);
  if ((threadIdx.x & 31) == 0) {
    unsigned long long* C4 = a.ctr + (size_t)r * 4;
    if (sa) atomicAdd(C4 + 1, (unsigned long long)sa);
    if (sc) atomicAdd(C4 + 2, (unsigned long long)sc);
    if (ss) atomicAdd(C4 + 3, (unsigned long long)ss);
  }
}

// Continuous update of a run's last day from the post-event counts, or the
// midpoint with the sums the stochastic step saved (earlier days' updates run in
// the next day's stochastic-step prologue).
__global__ void __launch_bounds__(kGenThreads) k_gen_cont(GenContArgs a) {
  __shared__ GenModelDev m;
  __shared__ GenRepParams p;
  const int r = blockIdx.y;
  grid_dependents_launch();
  copy16(&m, a.model, (int)(sizeof(GenModelDev) / 16));
  copy16(&p, a.params + r, (int)(sizeof(GenRepParams) / 16));
  __syncthreads();
  grid_dependency_wait();
  const int v = blockIdx.x * blockDim.x + threadIdx.x, N = a.N, nc = m.nc, ny = m.ny;
  if (v >= N) return;
  const int32_t* X = a.counts + (size_t)r * nc * N + v;
  double* Y = a.y + (size_t)r * ny * N + v;
  for (int q = 0; q < ny; ++q) {
    double U = u2d_exact(mask_sum(X, N, m.num[q], nc));
    double D = u2d_exact(mask_sum(X, N, m.den[q], nc));
    if (m.y_source == kGenYMidpoint) {
      const double* M = a.mid + ((size_t)r * ny + q) * 2 * N + v;
      U = __dmul_rn(0.5, __dadd_rn(M[0], U));
      D = __dmul_rn(0.5, __dadd_rn(M[N], D));
    }
    Y[(size_t)q * N] = gen_y_next(m, p, q, a.day, Y[(size_t)q * N], U, D);
  }
}

}  // namespace

size_t gen_ssa_smem_bytes(int nc, int nt) {
  return sizeof(GenModelDev) + sizeof(GenRepParams) + kGenThreads * sizeof(double) +
         (size_t)2 * nt * kGenThreads * sizeof(double) +
         (size_t)(kGenThreads / 32) * (32 / 8) * kGenMaxComp * sizeof(int32_t) + kGenThreads * sizeof(int32_t) +
         (size_t)nc * kGenThreads * sizeof(int32_t);
}

namespace {

size_t gen_f32_smem_bytes(int nc, int nt, int L, int tab16, int xrows) {
  return sizeof(GenModelDev) + (size_t)tab16 * 16 + kGenThreads * sizeof(double) +
         (size_t)2 * nt * kGenThreads * sizeof(double) +
         (size_t)(kGenThreads / kGenSeg) * (kGenMaxComp + L + xrows) * 4 + kGenThreads * sizeof(int32_t) +
         (size_t)(xrows + nc) * kGenThreads * 4;
}

using GenSsaKernel = void (*)(GenSsaArgs);
GenSsaKernel gen_ssa_kernel(int L) {
  return L == 4 ? k_gen_ssa<4> : L == 8 ? k_gen_ssa<8> : L == 16 ? k_gen_ssa<16> : k_gen_ssa<32>;
}

using GenEventsKernel = void (*)(GenEvArgs);
GenEventsKernel gen_events_kernel(int nc) {
  return nc <= kGenSmall ? k_gen_events_small<kGenSmall> : k_gen_events;
}

}  // namespace

// Transitions the kernel is unrolled for: the power of two that holds the model's.
int gen_unroll(int nt) {
  int L = 4;
  while (L < nt) L *= 2;
  return L;
}

// The limit belongs to the kernel, which every handle of its unrolled size shares: it is
// raised to what the device allows, never to one handle's own need, so that no handle
// lowers it for another.
static cudaError_t allow_smem(const void* k) {
  int dev = 0, most = 0;
  cudaFuncAttributes fa;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&most, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, k);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, most - (int)fa.sharedSizeBytes);
  return e;
}

cudaError_t gen_ssa_prepare(int nc, int nt, int L, int tab16, int xrows, int* blocks_per_sm) {
  const GenSsaKernel k = gen_ssa_kernel(L);
  const size_t smem = gen_f32_smem_bytes(nc, nt, L, tab16, xrows);
  cudaError_t e = allow_smem((const void*)k);
  if (e == cudaSuccess) e = allow_smem((const void*)k_gen_ssa_exact);
  if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, (const void*)k, kGenThreads, smem);
  return e;
}

cudaError_t launch_gen_ssa(GenSsaArgs a, int nt, int nc, cudaStream_t st) {
  if (!a.clock_margin) {
    a.warp_blocks = (a.n_big + kGenWarps - 1) / kGenWarps;
    const int per_block = kGenWarps * (32 / kGenSeg);
    a.group_blocks = (a.n_mid + per_block - 1) / per_block;
    const int rest = a.N - a.n_big - a.n_mid;
    const dim3 grid((unsigned)(a.warp_blocks + a.group_blocks + (rest + kGenThreads - 1) / kGenThreads), (unsigned)a.R);
    return launch_maybe_pdl(k_gen_ssa_exact, grid, dim3(kGenThreads), gen_ssa_smem_bytes(nc, nt), st, true, a);
  }
  // resident grid, fewer blocks when the units do not fill it (one unit a warp)
  const int64_t per = 32 / kGenSeg;
  const int64_t units =
      (int64_t)a.R * (a.n_big + ((int64_t)a.n_mid + per - 1) / per + ((int64_t)a.N - a.n_big - a.n_mid + 31) / 32);
  const int64_t grid = std::min<int64_t>(a.resident_blocks, (units + kGenWarps - 1) / kGenWarps);
  return launch_maybe_pdl(gen_ssa_kernel(a.L), dim3((unsigned)std::max<int64_t>(grid, 1)), dim3(kGenThreads),
                          gen_f32_smem_bytes(nc, nt, a.L, a.tab16, a.xrows), st, true, a);
}

cudaError_t launch_gen_events(const GenEvArgs& a, int nc, cudaStream_t st) {
  if (a.ncomp <= 0) return cudaSuccess;
  // a warp per component up to kGenEventWarps warps, then up to 32 per warp
  const int warps = std::max((a.ncomp + 31) / 32, std::min(a.ncomp, kGenEventWarps));
  const dim3 grid((unsigned)((warps + kGenWarps - 1) / kGenWarps), (unsigned)a.R);
  return launch_maybe_pdl(gen_events_kernel(nc), grid, dim3(kGenThreads), 0, st, true, a);
}

cudaError_t launch_gen_cont(const GenContArgs& a, cudaStream_t st) {
  const dim3 grid((unsigned)((a.N + kGenThreads - 1) / kGenThreads), (unsigned)a.R);
  return launch_maybe_pdl(k_gen_cont, grid, dim3(kGenThreads), 0, st, true, a);
}

}  // namespace episim
