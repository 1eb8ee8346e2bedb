// The residual step of a sweep (Eq. 5.11), run by one block per member.  A sweep's own
// step rides in the inverse y pass that follows the Green pass: nothing before the next
// sweep reads its result, so a block of that pass does it while the others transform.
// As a kernel of its own it took 5-8 us of FP64 latency and a launch between two passes
// (20-25% of a 64^3 sweep).
#pragma once
#include "kernels.h"

#include <cmath>

namespace bfcs {

// Member m's step; all threads of a block (at least one warp; threads past the last whole
// warp add nothing).  Sums the Green pass's partials in a fixed order for the block size.  r = sqrt(sum) / D, D = ||b_hat|| +
// xi_min |sigma_hat(0)|_F with sigma_hat(0) = N C0 E + tau_hat(0) and xi_min = 2 pi / max N_a.
//
// The step is one chain of latencies (an FP64 add takes 64 clocks, a square root or a
// division 600), and a small grid's y pass is no longer than it: the partials are
// requested before anything else is looked at, the normaliser and its reciprocal are
// formed by another warp beside the sum, and the warps' sums are added by shuffles.
static __device__ __noinline__ void resid_step(const ResidArgs& a, int m) {
  __shared__ double red[32];
  __shared__ double den_s, iden_s;
  IterState* st = a.sts + m;
  const ResidSlot* part = a.part + (long long)m * a.nparts;
  const int tid = threadIdx.x, nthr = blockDim.x & ~31, nw = nthr >> 5;
  const bool sweep_mode = a.mode == GM_SWEEP;
  const int seen = sweep_mode ? st->seen : 0;   // (written by the Green pass: the block's threads agree)
  const int sweep = st->iters, nc = st->next_check;
  double acc = 0.0;
  if (tid < nthr) {
#pragma unroll 4
    for (int i = tid; i < a.nparts; i += nthr) acc += part[i].num;
  }
  if (seen) return;
  if (tid == 0 && sweep_mode && a.io != nullptr) {
    // what the Green pass of this sweep moved besides its fixed traffic: d_prev read, d written
    const bool rd = a.check_max <= 1 || sweep == nc;
    const bool wr = a.check_max <= 1 || rd || sweep + 1 == nc || sweep + 1 >= st->maxit;
    atomicAdd(a.io, (unsigned long long)rd);
    atomicAdd(a.io + 1, (unsigned long long)wr);
  }
  const bool no_check = sweep_mode && a.check_max > 1 && sweep != nc;
  if (no_check) {
    // no residual on this sweep (the Green pass wrote no partials)
    __syncthreads();         // every thread has read the counters
    if (tid == 0) {
      if (sweep < a.hist_cap && a.hist != nullptr) a.hist[(long long)m * a.hist_cap + sweep] = NAN;
      st->iters = sweep + 1;
    }
    return;
  }
  if (tid == (nw > 1 ? nthr - 32 : 0)) {   // the normaliser, beside the sum
    const double* E = a.mem[m].E;
    const double trE = E[0] + E[1] + E[2];
    double s0[6];
    for (int c = 0; c < 6; ++c)
      s0[c] = a.n * (2.0 * a.mu0 * E[c] + (c < 3 ? a.lam0 * trE : 0.0)) + st->tau0[c];
    const double s0n = sqrt((s0[0] * s0[0] + s0[1] * s0[1]) + s0[2] * s0[2] +
                            2.0 * ((s0[3] * s0[3] + s0[4] * s0[4]) + s0[5] * s0[5]));
    const double den = st->bden + a.ximin * s0n;
    den_s = den;
    iden_s = 1.0 / den;
  }
  if (tid < nthr) {
    for (int off = 16; off > 0; off >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, off);
    if ((tid & 31) == 0) red[tid >> 5] = acc;
  }
  __syncthreads();
  if (tid >= 32) return;
  double t = tid < nw ? red[tid] : 0.0;
  for (int off = 16; off > 0; off >>= 1) t += __shfl_down_sync(0xffffffffu, t, off);
  if (tid != 0) return;
  const int warm = a.mem[m].warm;
  const double tol = st->tol;
  double r = sqrt(t);
  if (den_s > 0.0) r *= iden_s;
  if (!sweep_mode) { st->resid_final = r; return; }
  const bool skip_check = warm && sweep == 0;
  if (skip_check) r = INFINITY;
  if (sweep < a.hist_cap && a.hist != nullptr) a.hist[(long long)m * a.hist_cap + sweep] = r;
  // sweep of the next evaluation: with sparse evaluation, where the contraction
  // rate between the last two evaluations predicts r <= tol (at most check_max
  // sweeps ahead; every check_max sweeps when tol = 0), else the next sweep
  int gap = 1;
  if (a.check_max > 1 && !skip_check) {
    if (!(tol > 0.0)) {
      gap = a.check_max;
    } else if (st->checks > 0 && sweep > st->last_check && r > tol && r < st->resid_last && r > 0.0) {
      const double rate = pow(r / st->resid_last, 1.0 / (double)(sweep - st->last_check));
      const double need = ceil(log(tol / r) / log(rate));
      gap = (int)fmin(fmax(need, 1.0), (double)a.check_max);
    }
  }
  st->next_check = sweep + gap;
  if (!skip_check) {
    st->last_check = sweep;
    st->checks += 1;
  }
  st->resid_last = r;
  st->iters = sweep + 1;
  if (skip_check) return;
  if (!(r == r && r < INFINITY)) { st->diverged = 1; st->done = 1; return; }
  if (r <= tol) { st->done = 1; return; }
  // stall: the residual did not drop by 10% over stall_window sweeps
  if (a.stall_window > 0) {
    if (st->stall_ref == 0.0) { st->stall_ref = r; st->stall_at = sweep; }
    else if (sweep - st->stall_at >= a.stall_window) {
      if (r > 0.9 * st->stall_ref) { st->stalled = 1; st->done = 1; }
      else { st->stall_ref = r; st->stall_at = sweep; }
    }
  }
}

}  // namespace bfcs
