// C entries to internal pieces of libpf.so for tests: kernels whose special
// cases no load step can be made to reach.
#include "pf_hier.h"

using namespace pf;

extern "C" {

// The fused FP32 CG product at the given point of a run (started at `start`
// products, `used` by now): p and q as it leaves them.
int probe_cg_product(pf_hierarchy* h, int level, const float* x, float* p, float* q, const float* r, const float* mi,
                     double beta, int start, int used) {
  CgCtrl c{};
  c.rz = 1.0;
  c.beta = beta;
  c.start = start;
  c.used = used;
  c.cg_max = 1000;
  if (cudaMemcpyAsync(h->ctrl, &c, sizeof c, cudaMemcpyHostToDevice, h->st) != cudaSuccess) return 1;
  const CgDirIn dir{r, mi, h->ctrl};
  if (elem_hessvec32_dot(h->geo[level], h->mat[level], x, p, q, h->ctrl, h->scratch.partials, h->scratch.counter,
                         h->etile_part, h->p_dev, dir, h->st) != cudaSuccess)
    return 2;
  return cudaStreamSynchronize(h->st) != cudaSuccess ? 3 : 0;
}

// Sends the hierarchy's subproblems of small levels to separate launches.
void probe_separate_launches(pf_hierarchy* h) { h->sub_ok = false; }
int probe_one_launch(pf_hierarchy* h) { return h->sub_ok ? 1 : 0; }

// Lets the grid barrier of the next one-launch subproblem wait for an arrival
// that no CTA makes, for at most `polls` polls.
int probe_stuck_barrier(pf_hierarchy* h, long long polls) {
  h->sub_spin_limit = polls;
  SubCtrl c{};
  if (cudaMemcpyAsync(&c, h->sub_ctl, sizeof c, cudaMemcpyDeviceToHost, h->st) != cudaSuccess) return 1;
  if (cudaStreamSynchronize(h->st) != cudaSuccess) return 2;
  c.base += 1;
  if (cudaMemcpyAsync(h->sub_ctl, &c, sizeof c, cudaMemcpyHostToDevice, h->st) != cudaSuccess) return 3;
  return cudaStreamSynchronize(h->st) != cudaSuccess ? 4 : 0;
}

// A copy of the level's stored Galerkin operator.
int probe_galerkin_stencil(pf_hierarchy* h, int level, float* out) {
  const size_t n = size_t(galerkin_stencil_count(h->geo[level]));
  if (!h->lv[level].gs) return 1;
  if (cudaMemcpyAsync(out, h->lv[level].gs, sizeof(float) * n, cudaMemcpyDeviceToDevice, h->st) != cudaSuccess) return 2;
  return cudaStreamSynchronize(h->st) != cudaSuccess ? 3 : 0;
}

// The one-launch subproblem of a level: min g.s + s.S s / 2 over lo <= s <= hi
// (S and mi FP32 or FP64); stats: CG products, restarts.
int probe_subproblem(pf_hierarchy* h, int level, int fp32, const void* S, const void* mi, const double* g,
                     const double* lo, const double* hi, double* s, int cg_max, int max_restarts, int* stats) {
  SubIn in{};
  in.stencil = S;
  in.fp32 = fp32 != 0;
  in.gr = g;
  in.lo = lo;
  in.hi = hi;
  in.mi = mi;
  in.s = s;
  in.work = h->sub_work;
  in.partials = h->sub_partials;
  in.bar = h->sub_bar;
  in.ctl = h->sub_ctl;
  in.delta = 1.0;
  in.cauchy_c = 0.01;
  in.spin_limit = h->sub_spin_limit;
  in.backtracks = 30;
  in.cg_max = cg_max;
  in.max_restarts = max_restarts;
  if (subproblem_coop(h->geo[level], in, h->st) != cudaSuccess) return 1;
  SubCtrl c{};
  if (cudaMemcpyAsync(&c, h->sub_ctl, sizeof c, cudaMemcpyDeviceToHost, h->st) != cudaSuccess) return 2;
  if (cudaStreamSynchronize(h->st) != cudaSuccess) return 3;
  stats[0] = c.used;
  stats[1] = c.restarts;
  return c.failed ? 4 : 0;
}

// Whether the level holds the FP64 stencil of the mixed mode's small levels.
int probe_small_stencil(pf_hierarchy* h, int level) { return h->lv[level].small ? 1 : 0; }

}  // extern "C"
