// Stopping rule of the basic and Eyre-Milton schemes for one (cell, load) pair, shared by the control
// kernel (hom_solver.cu) and the on-chip solver of small grids (hom_resident2d.cu).
#pragma once

#include <cmath>

#include "hom_solve_args.cuh"

namespace hom {
namespace {

// Called by a whole warp whose lane k holds total k: the NC stress sums, the residual sum, the normalised
// residual sum and the compatibility residual sum (Eyre-Milton scheme) of iterate `it` over nv voxels.
// The scalar FP64 chain (square roots and divisions, hundreds of cycles each) runs side by side in the
// lanes.  Writes the pair's mean stress, errors and, where it stops, its status; lane 0 gets 1 if the
// pair stays active.
template <int NC>
__device__ __forceinline__ int control_pair(const SolveArgs& A, int pair, double nv, double sum, int it) {
  const int lane = threadIdx.x & 31;
  const bool em = A.partE != nullptr;
  int still = 0;
  double den2 = 0.0, e2 = 0.0;
#pragma unroll
  for (int k = 0; k < NC; ++k) {
    const double x = __shfl_sync(0xffffffffu, sum, k);
    den2 += x * x;
  }
  if (em) {
    const double* Ep = A.E + (size_t)pair * NC;
    for (int k = 0; k < NC; ++k) e2 += Ep[k] * Ep[k];
  }
  // An iterate clearly above the tolerance whose errors nobody reads goes on without a square root or a
  // division (the FP64 chain took 2-3 us of every iteration).
  if (A.quiet && it < A.max_iter) {
    const double q = __shfl_sync(0xffffffffu, sum, A.criterion == HOM_CRIT_E ? NC : NC + 1);
    const double c2 = em ? __shfl_sync(0xffffffffu, sum, NC + 2) : 0.0;
    const double t2 = (A.tol > 0.0 ? A.tol * A.tol : 0.0) * (1.0 + 1e-9);
    if (den2 > 0.0 && isfinite(den2) && isfinite(q) && isfinite(c2) && (q > t2 * den2 || c2 > t2 * (nv * nv) * e2))
      return lane == 0;
  }
  // lanes 0 .. NC - 1: the mean stress; NC and NC + 1: e and e_n; NC + 2: e_c
  double num = sum, den = nv;
  if (lane >= NC && lane < NC + 3) {
    if (A.res0 && lane < NC + 2) {  // adjoint: relative to the first iterate's residual
      double* r0 = A.res0 + 2 * pair + (lane - NC);
      if (it == 0) *r0 = sum;
      den = *r0;
      num = den > 0.0 ? sum / den : 0.0;
      den = 1.0;
    } else if (lane < NC + 2) {
      den = den2;
    } else {
      den = e2;
    }
    num = sqrt(num);
    den = sqrt(den) * (lane == NC + 2 ? nv : 1.0);
  }
  const double q = num / den;
  if (lane < NC) A.mean_sigma[(size_t)pair * NC + lane] = q;
  const double e = __shfl_sync(0xffffffffu, q, NC), en = __shfl_sync(0xffffffffu, q, NC + 1),
               ec = __shfl_sync(0xffffffffu, q, NC + 2);
  if (lane == 0) {
    A.err[pair] = e;
    A.errn[pair] = en;
    double crit = A.criterion == HOM_CRIT_E ? e : en;
    if (em) {  // Eyre-Milton: e_c = |eps_hat - P eps_hat| / (N_v |E|) must pass too
      A.errc[pair] = ec;
      crit = fmax(crit, ec);
      if (!isfinite(ec)) crit = ec;
    }
    int st = -1;
    const bool skip = A.warm && it == 0;  // warm start: g of the caller's field is unknown
    if (A.hist && !A.inner && it <= A.max_iter)
      A.hist[(size_t)pair * (A.max_iter + 1) + it] = skip ? (double)NAN : crit;
    if (A.inner) {  // defect-correction inner solve: a fixed number of iterations, no error test
      if (it >= A.kinner[pair]) st = HOM_STATUS_MAX_ITER;
    } else if (skip) {
      if (it >= A.max_iter) st = HOM_STATUS_MAX_ITER;
    } else if (!isfinite(crit)) st = HOM_STATUS_DIVERGED;
    else if (crit < A.tol) st = HOM_STATUS_CONVERGED;
    else if (it >= A.max_iter) st = HOM_STATUS_MAX_ITER;
    else {
      if (A.diverge_window > 0) {
        int gcount = crit > A.last_err[pair] ? A.grow[pair] + 1 : 0;
        A.grow[pair] = gcount;
        if (gcount >= A.diverge_window) st = HOM_STATUS_DIVERGED;
      }
      // stagnation: no new smallest error for stall_window iterations (the FP32 floor)
      if (st < 0 && A.stall_window > 0) {
        if (crit < A.best_err[pair]) {
          A.best_err[pair] = crit;
          A.best_it[pair] = it;
        } else if (it - A.best_it[pair] >= A.stall_window) {
          st = HOM_STATUS_STALLED;
        }
      }
    }
    if (!skip) A.last_err[pair] = crit;
    if (st >= 0) {
      A.status[pair] = st;
      A.iters[pair] = it;
      A.active[pair] = 0;
    } else {
      still = 1;
    }
  }
  return still;
}

}  // namespace
}  // namespace hom
