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
static __device__ __noinline__ void resid_step(const ResidArgs& a, int m) {
  __shared__ double red[32];
  __shared__ double den_s;
  __shared__ int no_check;   // decided by one thread: thread 0 advances st->iters below
  IterState* st = a.sts + m;
  if (a.mode == GM_SWEEP && st->seen) return;   // (written by the Green pass: the block's threads agree)
  if (threadIdx.x == 0) {
    const int sw = st->iters, nc = st->next_check;
    no_check = a.mode == GM_SWEEP && a.check_max > 1 && sw != nc;
    if (a.io != nullptr && a.mode == GM_SWEEP) {
      // what the Green pass of this sweep moved besides its fixed traffic: d_prev read, d written
      const bool rd = a.check_max <= 1 || sw == nc;
      const bool wr = a.check_max <= 1 || rd || sw + 1 == nc || sw + 1 >= a.maxit;
      atomicAdd(a.io, (unsigned long long)rd);
      atomicAdd(a.io + 1, (unsigned long long)wr);
    }
  }
  __syncthreads();
  if (no_check) {
    // no residual on this sweep (the Green pass wrote no partials)
    if (threadIdx.x == 0) {
      const int sweep = st->iters;
      if (sweep < a.hist_cap && a.hist != nullptr) a.hist[(long long)m * a.hist_cap + sweep] = NAN;
      st->iters = sweep + 1;
    }
    return;
  }
  const int nthr = blockDim.x & ~31, nw = nthr >> 5;
  if (threadIdx.x == (nw > 1 ? 32 : 0)) {   // the normaliser, beside the sum
    const double* E = a.mem[m].E;
    const double trE = E[0] + E[1] + E[2];
    double s0[6];
    for (int c = 0; c < 6; ++c)
      s0[c] = a.n * (2.0 * a.mu0 * E[c] + (c < 3 ? a.lam0 * trE : 0.0)) + st->tau0[c];
    const double s0n = sqrt(s0[0] * s0[0] + s0[1] * s0[1] + s0[2] * s0[2] +
                            2.0 * (s0[3] * s0[3] + s0[4] * s0[4] + s0[5] * s0[5]));
    den_s = st->bden + 6.283185307179586 / (double)a.maxdim * s0n;
  }
  const ResidSlot* part = a.part + (long long)m * a.nparts;
  if ((int)threadIdx.x < nthr) {
    double acc = 0.0;
#pragma unroll 4
    for (int i = threadIdx.x; i < a.nparts; i += nthr) acc += part[i].num;
    for (int off = 16; off > 0; off >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, off);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
  }
  __syncthreads();
  if (threadIdx.x != 0) return;
  double t = 0.0;
  for (int w = 0; w < nw; ++w) t += red[w];
  const double den = den_s;
  const int warm = a.mem[m].warm;
  const double tol = a.mem[m].tol >= 0.0 ? a.mem[m].tol : a.tol;
  double r = den > 0.0 ? sqrt(t) / den : sqrt(t);
  if (a.mode == GM_FINAL) { st->resid_final = r; return; }
  const int sweep = st->iters;
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
