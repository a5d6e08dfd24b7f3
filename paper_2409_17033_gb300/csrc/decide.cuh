// The SP2 branch and stop decision of one step (Eq. DM0 with the readings of
// the stop rule in sp2.h): one block of threads reduces the step's trace
// partials in a fixed order and one thread updates the device state. Shared by
// the decision kernel and by the squares whose last block takes it: on the CUDA cores, by
// digits, and on the tensor cores with tiles below 256 columns.
#pragma once
#include "sp2_internal.h"

namespace sp2 {
namespace {

constexpr int kStall = 4;  // steps without a new minimum of f that mark the precision floor

__device__ double block_sum(double v) {
  __shared__ double red[32];
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  __syncthreads();
  if (l == 0) red[w] = v;
  __syncthreads();
  int nw = (blockDim.x + 31) >> 5;
  v = (threadIdx.x < nw) ? red[threadIdx.x] : 0.0;
  if (w == 0)
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;  // valid in thread 0
}

// Tells the host of the step: one 8-byte word (token and whether the recursion goes
// on). Only at its end (a stop, an abort, the last step) the other fields go out
// first, with a system-wide fence between, which waits for the host's memory.
__device__ __forceinline__ void post_snapshot(const DevState* st, const DecideParams& p,
                                              int stop_at) {
  if (!p.snap) return;
  volatile HostSnap* s = p.snap;
  const int ab = *((volatile const int*)&st->abort_flag);
  const int last = p.n - 1 >= (p.fixed_m > 0 ? p.fixed_m : p.max_iter);
  const unsigned long long end = stop_at != 0 || ab || last ? 1ull : 0ull;
  if (end) {
    s->stop_at = stop_at;
    s->nonfinite = st->nonfinite;
    s->abort_flag = ab;
    s->backtracked = st->backtracked;
    s->stop_step = st->stop_step;
    s->bounds[0] = st->bounds[0];
    s->bounds[1] = st->bounds[1];
    s->alpha = st->alpha;
    s->beta = st->beta;
    s->work_kblocks = st->work_kblocks;
    __threadfence_system();
  }
  s->word = 2ull * p.token + end;
}

// three block-wide sums at once, each in block_sum's order
__device__ void block_sum3(double& a, double& b, double& c) {
  __shared__ double red3[3][32];
  for (int o = 16; o > 0; o >>= 1) {
    a += __shfl_xor_sync(0xffffffffu, a, o);
    b += __shfl_xor_sync(0xffffffffu, b, o);
    c += __shfl_xor_sync(0xffffffffu, c, o);
  }
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  __syncthreads();
  if (l == 0) {
    red3[0][w] = a;
    red3[1][w] = b;
    red3[2][w] = c;
  }
  __syncthreads();
  if (w != 0) return;
  const int nw = (blockDim.x + 31) >> 5;
  a = l < nw ? red3[0][l] : 0.0;
  b = l < nw ? red3[1][l] : 0.0;
  c = l < nw ? red3[2][l] : 0.0;
  for (int o = 16; o > 0; o >>= 1) {
    a += __shfl_xor_sync(0xffffffffu, a, o);
    b += __shfl_xor_sync(0xffffffffu, b, o);
    c += __shfl_xor_sync(0xffffffffu, c, o);
  }   // valid in thread 0
}

// One thread's part of the decision: everything it needs of earlier steps is read
// at once, beside the partials (one memory latency instead of a chain of them).
struct DecideHist {
  int stop_at, nbest, plane, sg1, sg2;
  double fbest, fold, f1, f2, f3, fk;   // f_{s-1}, f_{s-2}, f_{s-3}, f_{s-kStall}
};

// Returns stop_at.
__device__ __forceinline__ int decide_one(DevState* st, const DecideParams& p, const DecideHist& h,
                                          double t1, double t2, double f) {
  if (h.stop_at != 0) return h.stop_at;  // already stopped: later steps are no-ops
  const int n = p.n;
  const int s = n - 1;  // the step that produced X_n (0 for X_1)
  st->t1[n] = t1;
  st->t2[n] = t2;
  if (n >= 2) st->f[n - 1] = f;  // the step that produced X_n measured X_{n-1}
  // split-tail mode: step n (X_n -> X_{n+1}) uses single-plane products while the
  // idempotency error of the last measured iterate exceeds tail_f; once a step
  // has used split products, every later one does
  if (p.tail_f > 0.0) st->plane1[n] = n == 1 ? 1 : (h.plane && f > p.tail_f ? 1 : 0);
  if (!isfinite(t1) || !isfinite(t2)) {
    st->nonfinite = 1;
    st->stop_at = (n - 1 >= 1) ? n - 1 : -1;
    return (n - 1 >= 1) ? n - 1 : -1;
  }
  // floor candidates: X_s (f known now) with f <= gate and the smallest f so far
  int nbest = h.nbest;
  if (p.fixed_m == 0 && p.floor_gate > 0.0 && s >= 2 && f <= p.floor_gate &&
      (nbest == 0 || f < h.fbest)) {
    nbest = s;
    st->fbest = f;
    st->nbest = s;
    st->keep_step = s;
  }
  if (p.fixed_m > 0) {
    if (s == p.fixed_m) st->stop_at = s;
    return s == p.fixed_m ? s : 0;  // branches preset by the host
  }
  // the smallest f of the steps before the last kStall
  double best = h.fold;
  if (s > kStall) {
    best = s - kStall == 1 ? h.fk : fmin(h.fold, h.fk);
    st->fold = best;
  }
  if (s >= 1 && s >= p.min_iter) {
    const double e = fabs(t1 - t2);
    bool stop = false, floor_stop = false;
    if (p.idem_tol > 0.0 && e <= p.idem_tol) stop = true;
    // precision floor on f (see the stop rule in sp2.h):
    //   opposite branches at steps s-2, s-1, f_{s-2} <= gate and f_s >= f_{s-2}; or
    //   min f_1..f_{s-STALL} <= gate and none of f_{s-STALL+1..s} below it
    if (!stop && p.floor_gate > 0.0) {
      if (s >= 3 && h.sg2 != h.sg1 && h.f2 <= p.floor_gate && f >= h.f2) floor_stop = true;
      // block-sparse recursion: from f <= 1e-4 a pair of opposite steps cuts f at
      // least 600-fold in exact arithmetic; less than twofold is the threshold's floor
      if (!floor_stop && p.ratio_floor && s >= 3 && h.sg2 != h.sg1 && h.f2 <= kRatioGate &&
          f >= 0.5 * h.f2)
        floor_stop = true;
      if (!floor_stop && s > kStall) {
        const double recent = fmin(fmin(fmin(h.f3, h.f2), h.f1), f);
        if (best <= p.floor_gate && recent >= best) floor_stop = true;
      }
      if (floor_stop) stop = true;
    }
    if (stop) {
      st->stop_step = s;
      // at the floor the result is the kept candidate X_nbest (M = nbest - 1 steps)
      const bool back = floor_stop && nbest >= 2 && nbest - 1 < s;
      if (back) st->backtracked = 1;
      st->stop_at = back ? nbest - 1 : s;
      return back ? nbest - 1 : s;
    }
  }
  // Eq. DM0 branch: the trace after X^2 is t2, after 2X - X^2 it is 2 t1 - t2.
  st->sigma[n] = (fabs(t2 - p.nocc) <= fabs(2.0 * t1 - t2 - p.nocc)) ? 1 : -1;
  return 0;
}

__device__ __forceinline__ void load_hist(const DevState* st, const DecideParams& p, DecideHist& h) {
  static_assert(kStall == 4, "the decision reads f of the last four steps");
  const int s = p.n - 1;
  h.stop_at = st->stop_at;
  h.nbest = st->nbest;
  h.fbest = st->fbest;
  h.fold = st->fold;
  h.plane = st->plane1[s >= 0 ? s : 0];
  h.sg1 = s >= 1 ? st->sigma[s - 1] : 0;
  h.sg2 = s >= 2 ? st->sigma[s - 2] : 0;
  h.f1 = s >= 1 ? st->f[s - 1] : 0.0;
  h.f2 = s >= 2 ? st->f[s - 2] : 0.0;
  h.f3 = s >= 3 ? st->f[s - 3] : 0.0;
  h.fk = s >= kStall ? st->f[s - kStall] : 0.0;
}

constexpr int kWarpParts = 512;   // up to this many partials one warp takes the decision

// The decision by the first warp of a block (every thread may call): few partials
// cost a whole block more in FP64 shuffles (64 clocks a warp and instruction) and
// barriers than one warp's additions take: 8 us at the end of a product against 2.
// Reads the partials with cache-global loads: they come from the other blocks of
// the same launch.
__device__ __noinline__ void decide_warp(const Part3* part, DevState* st, const DecideParams& p) {
  if (threadIdx.x >= 32) return;
  DecideHist h;
  load_hist(st, p, h);
  double t1 = 0.0, t2 = 0.0, f = 0.0;
  for (int i = threadIdx.x; i < p.nparts; i += 32) {
    t1 += __ldcg(&part[i].t1);
    t2 += __ldcg(&part[i].t2);
    f += __ldcg(&part[i].f);
  }
  for (int o = 16; o > 0; o >>= 1) {
    t1 += __shfl_xor_sync(0xffffffffu, t1, o);
    t2 += __shfl_xor_sync(0xffffffffu, t2, o);
    f += __shfl_xor_sync(0xffffffffu, f, o);
  }
  if (threadIdx.x != 0) return;
  const int stop_at = decide_one(st, p, h, t1, t2, f);
  post_snapshot(st, p, stop_at);
}

// The same by a whole block (every thread calls).
__device__ __noinline__ void decide_block(const Part3* part, DevState* st, const DecideParams& p) {
  if (p.nparts <= kWarpParts) {
    decide_warp(part, st, p);
    return;
  }
  DecideHist h;
  if (threadIdx.x == 0) load_hist(st, p, h);
  double t1 = 0.0, t2 = 0.0, f = 0.0;
  for (int i = threadIdx.x; i < p.nparts; i += blockDim.x) {
    t1 += __ldcg(&part[i].t1);
    t2 += __ldcg(&part[i].t2);
    f += __ldcg(&part[i].f);
  }
  block_sum3(t1, t2, f);
  if (threadIdx.x != 0) return;
  const int stop_at = decide_one(st, p, h, t1, t2, f);
  post_snapshot(st, p, stop_at);
}

// After the decision, by the same block: X_s into the candidate's place when step s made
// it the best so far. Only a few steps do, near the end, and a launch of its own for
// every step (k_keep_best) took 2 us of a small step: FP64 density at N = 128 590 -> 550
// us. One block copies 128 KB in some 8 us but 1 MB in 17 (BF16X2 at N = 300, where a
// recursion has more candidates, 783 -> 850 us), and in the larger products' kernels
// this code costs registers (FP32 forward chi at N = 1500 5 % slower): the small FP64
// square alone has it, up to kKeepSmall.
__device__ __forceinline__ void keep_candidate(const DevState* st, const DecideParams& p) {
  if (p.keep_n == 0) return;
  __syncthreads();
  if (*((volatile const int*)&st->keep_step) != p.n - 1) return;
  const uint4* src = static_cast<const uint4*>(p.keep_src);
  uint4* dst = static_cast<uint4*>(p.keep_dst);
  constexpr int U = 8;
  for (int i0 = threadIdx.x; i0 < p.keep_n; i0 += U * blockDim.x) {
    uint4 v[U];
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (i0 + u * (int)blockDim.x < p.keep_n) v[u] = src[i0 + u * blockDim.x];
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (i0 + u * (int)blockDim.x < p.keep_n) dst[i0 + u * blockDim.x] = v[u];
  }
}

// The end of a square: its last block takes the step decision (every thread of every
// block calls, its partials stored). KEEP: and keeps a small candidate.
// nblocks: how many blocks call (0: the whole grid).
template <bool KEEP = false>
__device__ __forceinline__ void last_block_decides(const Part3* part, const SimtDecide& dec,
                                                   unsigned nblocks = 0) {
  __shared__ int last;
  if (threadIdx.x == 0) {
    __threadfence();
    last = atomicAdd(dec.done, 1u) == (nblocks ? nblocks : gridDim.x) - 1;
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  decide_block(part, dec.st, dec.p);
  if (threadIdx.x == 0) *dec.done = 0u;
  if constexpr (KEEP) keep_candidate(dec.st, dec.p);
}

}  // namespace
}  // namespace sp2
