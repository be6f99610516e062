// Ends of the kernels that carry a PCG reduction: the block sums go to the
// partials, and the last block forms the CG scalars and flags.
#pragma once

#include "mfg_internal.cuh"
#include "reduce.cuh"

namespace mfg {

// After q = AAt p: acc = this thread's share of p.q; alpha = rz / (p.q).
__device__ __forceinline__ void aat_tail(double acc, double* partials, DevScalars* sc) {
  double part[1] = {acc};
  block_sum<1>(part);
  if (!publish_and_check_last<1>(part, partials, &sc->counter)) return;
  double tot[1];
  gather_partials<1>(partials, tot);
  if (flat_tid() == 0) {
    sc->pq = tot[0];
    if (tot[0] > 0.0 && isfinite(tot[0])) {
      sc->alpha = sc->rz / tot[0];
    } else {
      sc->alpha = 0.0;
      sc->cg_done = 1;
      if (sc->status == MFG_OK) sc->status = MFG_ERR_NONFINITE;
    }
    sc->counter = 0;
  }
}

// After z += alpha p, r -= alpha q: rr = this thread's share of ||r||^2; the
// convergence test.
__device__ __forceinline__ void zr_tail(double rr, double* partials, DevScalars* sc) {
  double part[1] = {rr};
  block_sum<1>(part);
  if (!publish_and_check_last<1>(part, partials, &sc->counter)) return;
  double tot[1];
  gather_partials<1>(partials, tot);
  if (flat_tid() == 0) {
    sc->rr = tot[0];
    sc->cg_it += 1;
    const double tol = sc->cg_tol;
    if (!isfinite(tot[0])) {
      sc->cg_done = 1;
      if (sc->status == MFG_OK) sc->status = MFG_ERR_NONFINITE;
    } else if (tot[0] <= tol * tol * sc->bnorm2) {
      sc->cg_done = 1;
    } else if (sc->cg_it >= sc->max_cg) {
      sc->cg_done = 1;
      if (sc->status == MFG_OK) sc->status = MFG_ERR_NOT_CONVERGED;
    }
    sc->counter = 0;
  }
}

// After zp = P^{-1} r: a0, a1 = this thread's shares of r.zp and q.zp; beta
// (Polak-Ribiere when flex, else Fletcher-Reeves).
__device__ __forceinline__ void dot_tail(double a0, double a1, int flex, double* partials, DevScalars* sc) {
  double part[2] = {a0, a1};
  block_sum<2>(part);
  if (!publish_and_check_last<2>(part, partials, &sc->counter)) return;
  double tot[2];
  gather_partials<2>(partials, tot);
  if (flat_tid() == 0) {
    const double rz_old = sc->rz;
    sc->qz = tot[1];
    sc->beta = flex ? (-sc->alpha * tot[1] / rz_old) : (tot[0] / rz_old);
    sc->rz = tot[0];
    if (!isfinite(sc->beta) || !(tot[0] > 0.0)) {
      sc->cg_done = 1;
      if (sc->status == MFG_OK) sc->status = MFG_ERR_NONFINITE;
    }
    sc->counter = 0;
  }
}

}  // namespace mfg
