// Device pieces of the FP32 projected-CG subproblem shared by its vector
// passes (pf_solver.cu) and the product's last pass (pf_kernels.cu).
#pragma once
#include "pf_internal.h"

namespace pf {

__device__ __forceinline__ double clampv(double x, double lo, double hi) {
  return fmin(fmax(x, lo), hi);
}
__device__ __forceinline__ float clampv(float x, float lo, float hi) {
  return fminf(fmaxf(x, lo), hi);
}

__device__ __forceinline__ bool is_free(float lo, float hi, float s) { return lo - s < 0.f && 0.f < hi - s; }

// Start of a CG run from a restart's (r.r, r.M^-1 r) on the device; a run that
// starts already converged is stopped before its first iteration (CG_CONV), so
// the host needs no read-back before it.
__device__ __forceinline__ void cg_start(CgCtrl* c, double rr, double rz) {
  c->rr = rr;
  c->rz = rz;
  c->alpha = 0.0;
  c->beta = 0.0;
  c->kappa = 0.0;
  c->start = c->used;
  c->no_search = 1;
  const bool stop = sqrt(rr) <= c->tol || rr == 0.0;
  c->done = stop ? 1 : 0;
  c->state = stop ? CG_CONV : CG_RUNNING;
}

// What a dof adds to the start of a CG run at s: r, p = M^-1 r and the sums
// (r.r, r.M^-1 r).
__device__ __forceinline__ void cg_init_lane(float lo, float hi, float s, float g, float hs, float m, float& r,
                                             float& p, float& rr, float& rz) {
  const float ri = is_free(lo, hi, s) ? -(g + hs) : 0.f;
  const float zi = m * ri;
  r = ri;
  p = zi;
  rr += ri * ri;
  rz += ri * zi;
}

// What a dof adds to the test of a projected step t with Ht = H t, and to the
// start of the CG run at t: (r.r, r.M^-1 r, g.t, t.Ht, (g + Hs).(t - s)).
__device__ __forceinline__ void cg_search_lane(float lo, float hi, float s, float hs, float t, float ht,
                                               float g, float m, float& r, float& p, float (&o)[5]) {
  o[2] += g * t;
  o[3] += t * ht;
  o[4] += (g + hs) * (t - s);
  cg_init_lane(lo, hi, t, g, ht, m, r, p, o[0], o[1]);
}

// The end of a projected search, from those sums: t accepted (s and t swap by
// the parity of restarts) and the next run started, or rejected.
__device__ __forceinline__ void cg_search_done(CgCtrl* c, const double (&v)[5], double cauchy_c) {
  c->searches += 1;
  c->no_search = 1;
  const double m_t = v[2] + 0.5 * v[3];
  if (!(m_t <= c->m_s + cauchy_c * v[4])) {
    c->done = 1;
    c->state = CG_REJECT;
    return;
  }
  c->m_s = m_t;
  c->restarts += 1;
  if (c->restarts > c->max_restarts || c->used >= c->cg_max) {
    c->done = 1;
    c->state = CG_STOP;
    return;
  }
  cg_start(c, v[0], v[1]);
}

}  // namespace pf
