// ctl.cuh -- control block of the device-driven solve and the decisions that
// the last block of a kernel takes inside its loops (graph.cu has the rest).
#pragma once

#include "common.cuh"

namespace plc {

// Per-context control block (device memory).
struct DevCtl {
  // options (written by ctl_init at every launch)
  double tol, mixed_switch, eta_max, step_cap, g0_opt;
  int max_newton, max_cg, mixed;
  // state
  double g0, prev_rel, f0, xg, scale, eps;
  int it, q, par, fp64, stop, status, loops, cg_count;
  int check;   // the FP32 gradient passed the stopping test at the switch
  // statistics
  long long cg_iters, grad_evals, grad_ffts, grad_ffts_fp64, kernels;
  double grad_rel, neg_logpost;
};

__device__ __forceinline__ double f_of(const DevScalars* sc) { return 0.5 * sc->red[0] + sc->red[1]; }
__device__ __forceinline__ double scale_of(const DevScalars* sc) {
  return (sc->red[1] + sc->red[3]) + sc->red[4] + fabs(f_of(sc));
}

// Conditional loop around a captured kernel; t null outside graphs.
struct LoopCtl {
  DevCtl* t;
  cudaGraphConditionalHandle h;
  int nk;                       // kernels of one pass of the loop's body
};

// End of a CG iteration: another one unless the CG is done or at its cap.
__device__ __forceinline__ void ctl_cg(const LoopCtl& c, int done) {
  if (!c.t) return;
  c.t->kernels += c.nk;
  c.t->cg_count += 1;
  cudaGraphSetConditional(c.h, (!done && c.t->cg_count < c.t->max_cg) ? 1 : 0);
}

// Armijo test of the trial just evaluated; accept (the trial's field set
// becomes current) or halve tau.  The 30th trial is accepted as it is.
__device__ __forceinline__ void ctl_ls(const LoopCtl& c, DevScalars* sc) {
  DevCtl* t = c.t;
  if (!t) return;
  t->kernels += c.nk;
  t->grad_evals += 1;
  const double f = f_of(sc), tau = sc->tau;
  const bool ok = f <= t->f0 + 1e-4 * tau * t->xg || -tau * t->xg < t->eps * t->scale || t->q >= 29;
  if (ok) {
    t->par ^= 1;
    t->it += 1;
  } else {
    sc->tau = 0.5 * tau;
    t->q += 1;
  }
  cudaGraphSetConditional(c.h, ok ? 0 : 1);
}

}  // namespace plc
