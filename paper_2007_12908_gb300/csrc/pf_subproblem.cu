// The trust-region subproblem of a small level (eq. model_qp, projected-search
// truncated CG) in one cooperative launch.
//
// On grids of a few thousand nodes a CG iteration is five short launches: the
// product, two reductions, the direction and the condition of the graph's
// while node, which itself costs 5.5 us a turn; every restart adds a
// read-back of 13 us per scalar.  A 65^2 FP64 load step took 34 to 37 ms for
// about 1,030 iterations, some 30 us each.  Here the whole solve -- Cauchy
// point, CG runs, projected searches, restarts -- is one kernel whose CTAs
// meet at a grid barrier: two per CG iteration, which takes 9.5 us (3.5 of them
// the barriers' latency, the rest FP64 chains: the product's 27 multiply-adds
// in 9 warps of an SM at 16 cycles each, the trees of the sums, a division),
// and the load step 13 ms.
//
// A row (node and field) belongs to one lane for the whole solve: its vectors
// stay in registers, and where they fit (all but FP64 in 3D) so do its stencil
// entries, shared by the three threads of the row's three lines of offsets.
// Only what neighbours read goes through memory: the direction p is formed
// where it is read, z + beta p_old from two published vectors, so that its
// update needs no barrier of its own.  Scalars are summed from one partial per
// CTA, by every CTA in the same order, so that all take the same branches; the
// FP64 arithmetic on them (divisions, square roots) runs in one thread of a
// CTA, because an FP64 instruction holds the SM's pipe for 16 cycles per warp
// (repeated in every warp, it took 8 us of an iteration).
//
// The launch is cooperative (every CTA resident), and every wait has an
// iteration limit after which the kernel raises `failed` and returns; the
// caller then solves the subproblem with separate launches.
#include <algorithm>
#include <cmath>

#include "pf_hier.h"
#include "pf_reduce.cuh"

namespace pf {

namespace {

constexpr int kLanes = 128, kLines = 3, kThreads = kLanes * kLines;
constexpr int kMaxCoopBlocks = 1216;       // partials hold this many

template <int D, class TS, class V>
struct SubArgs {
  Geom g;
  int rows;                    // rows per CTA, at most kLanes
  const TS* S;
  const double *gr, *lo, *hi;  // FP64 model gradient and box (rounded to V here)
  const V* mi;                 // Jacobi inverse, or null
  double* s;                   // the step (FP64)
  V *b0, *b1, *z, *pa, *pb;    // published vectors
  double* partials;            // 2 x 4 x kMaxCoopBlocks
  unsigned* bar;               // arrivals so far
  SubCtrl* ctl;
  double delta, cauchy_c;
  long long spin_limit;
  int backtracks, cg_max, max_restarts;
};

__device__ __forceinline__ double box_lo(double v, double) { return v; }
__device__ __forceinline__ double box_hi(double v, double) { return v; }
// the FP32 box lies inside the FP64 one (lo <= 0 <= hi)
__device__ __forceinline__ float box_lo(double v, float) { return __double2float_ru(v); }
__device__ __forceinline__ float box_hi(double v, float) { return __double2float_rd(v); }
__device__ __forceinline__ double clamp_v(double x, double lo, double hi) { return fmin(fmax(x, lo), hi); }
__device__ __forceinline__ float clamp_v(float x, float lo, float hi) { return fminf(fmaxf(x, lo), hi); }
__device__ __forceinline__ double fma_v(double a, double b, double c) { return fma(a, b, c); }
__device__ __forceinline__ float fma_v(float a, float b, float c) { return fmaf(a, b, c); }

template <int D, class TS, class V, bool CACHE>
struct Sub {
  static constexpr int F = D + 1, NK = D == 3 ? 9 : 3;  // offsets of a line of threads
  const SubArgs<D, TS, V>& A;
  int lane, line, nb;
  long long row;
  bool live, owner;
  int turn = 0;          // barriers passed (partials alternate)
  unsigned target;       // thread 0: arrivals that open the next barrier
  // scalars of the solve, kept by thread 0 and read by all
  struct Shared {
    V part[kLines][kLanes];
    double val[3][kLanes], res[4];
    int go;
    double t, tt1, k1, m_s, tol, tol2, rz;
    V tt, alpha, beta, amax;
    int state, have, used;
  };
  Shared& sh;
  TS a[CACHE ? NK : 1][F];
  unsigned in = 0;       // neighbours inside the grid
  long long off0;        // first neighbour's offset from the node
  const TS* s0;
  long long node;

  __device__ Sub(const SubArgs<D, TS, V>& args, Shared& shared) : A(args), sh(shared) {
    target = A.ctl->base;  // the counter's value when every earlier launch had ended
    lane = threadIdx.x % kLanes;
    line = threadIdx.x / kLanes;
    nb = gridDim.x;
    row = blockIdx.x * (long long)A.rows + lane;
    live = lane < A.rows && row < (long long)F * A.g.N;
    owner = live && line == 0;
    const long long r = live ? row : 0;
    const int f = int(r / A.g.N);
    node = r - (long long)f * A.g.N;
    const int ix = int(node % A.g.n[0]);
    const int iy = int((node / A.g.n[0]) % A.g.n[1]);
    const int iz = D == 3 ? int(node / ((long long)A.g.n[0] * A.g.n[1])) : 0;
    // line: the y offset in 2D (3 entries along x), the z offset in 3D (9)
    const int d = line - 1;
#pragma unroll
    for (int k = 0; k < NK; ++k) {
      const int dx = k % 3 - 1, dy = D == 3 ? k / 3 - 1 : d, dz = D == 3 ? d : 0;
      const bool ok = ix + dx >= 0 && ix + dx < A.g.n[0] && iy + dy >= 0 && iy + dy < A.g.n[1] &&
                      iz + dz >= 0 && iz + dz < A.g.n[2];
      if (ok) in |= 1u << k;
    }
    off0 = D == 3 ? d * (long long)A.g.n[0] * A.g.n[1] : d * (long long)A.g.n[0];
    s0 = A.S + ((long long)line * NK * F + f) * F * A.g.N + node;
    if constexpr (CACHE)
#pragma unroll
      for (int k = 0; k < NK; ++k)
#pragma unroll
        for (int h = 0; h < F; ++h) a[k][h] = s0[(long long)(k * F * F + h) * A.g.N];
  }

  // This row of S times the published vector b, or times z + beta b where z
  // is given; the result is the owner's.
  __device__ V product(const V* b, const V* z, V beta) {
    // whole warps without a row skip the arithmetic (their partial sums are
    // not read)
    if (!__any_sync(0xffffffffu, live)) {
      __syncthreads();
      return V(0);
    }
    V acc[F];
#pragma unroll
    for (int h = 0; h < F; ++h) acc[h] = V(0);
#pragma unroll
    for (int k = 0; k < NK; ++k) {
      const int dx = k % 3 - 1, dy = D == 3 ? k / 3 - 1 : 0;
      const bool ok = (in >> k) & 1;
      const long long j = ok ? node + off0 + dx + dy * (long long)A.g.n[0] : node;
#pragma unroll
      for (int h = 0; h < F; ++h) {
        V v = __ldcg(b + h * A.g.N + j);
        if (z) v = fma_v(beta, v, __ldcg(z + h * A.g.N + j));
        const TS e = CACHE ? a[CACHE ? k : 0][h] : s0[(long long)(k * F * F + h) * A.g.N];
        acc[h] += V(e) * (ok ? v : V(0));
      }
    }
    V sum = (acc[0] + acc[1]) + (F == 4 ? acc[2] + acc[F - 1] : acc[2]);
    if (line > 0) sh.part[line][lane] = sum;
    __syncthreads();
    if (line == 0) sum += sh.part[1][lane] + sh.part[2][lane];
    return sum;
  }

  // Grid barrier on a counter that only grows; false once a wait has run out
  // anywhere.
  __device__ bool barrier() {
    __syncthreads();
    if (threadIdx.x == 0) {
      sh.go = 1;
      target += unsigned(nb);
      asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(A.bar) : "memory");
      long long spin = 0;
      for (;;) {
        unsigned c;
        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(c) : "l"(A.bar) : "memory");
        if (int(c - target) >= 0) break;
        ++spin;
        if ((spin & 255) == 0 && (spin > A.spin_limit || *(volatile int*)&A.ctl->failed)) {
          atomicExch(&A.ctl->failed, 1);
          sh.go = 0;
          break;
        }
      }
    }
    __syncthreads();
    ++turn;
    return sh.go != 0;
  }

  // Sums of K values over all owners (the first with Op0), also making this
  // CTA's published values visible to all; thread 0 passes them to fin, whose
  // results in sh every thread may read afterwards.
  template <int K, class Op0 = OpSum, class Fin>
  __device__ bool sums(const double (&v)[K], Fin fin) {
    double* p = A.partials + (turn & 1) * 4 * kMaxCoopBlocks;
    const int wl = threadIdx.x & 31, w = threadIdx.x >> 5;
    // one warp combines each value (see block_reduce)
    if (w < kLanes / 32)
#pragma unroll
      for (int k = 0; k < K; ++k) sh.val[k][threadIdx.x] = owner ? v[k] : (k == 0 ? Op0::id() : 0.0);
    __syncthreads();
    if (w < K) {
      double x = sh.val[w][wl];
#pragma unroll
      for (int i = 32; i < kLanes; i += 32) x = w == 0 ? Op0::op(x, sh.val[w][wl + i]) : x + sh.val[w][wl + i];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        const double y = __shfl_xor_sync(0xffffffffu, x, o);
        x = w == 0 ? Op0::op(x, y) : x + y;
      }
      if (wl == 0) p[w * kMaxCoopBlocks + blockIdx.x] = x;
    }
    if (!barrier()) return false;
    if (w < K) {
      const double id = w == 0 ? Op0::id() : 0.0;
      double x = id;
      for (int b0 = wl; b0 < nb; b0 += 32 * 5) {  // one round of loads for 160 CTAs
        double y[5];
#pragma unroll
        for (int i = 0; i < 5; ++i) {
          const int b = b0 + 32 * i;
          y[i] = b < nb ? __ldcg(p + w * kMaxCoopBlocks + b) : id;
        }
#pragma unroll
        for (int i = 0; i < 5; ++i) x = w == 0 ? Op0::op(x, y[i]) : x + y[i];
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        const double y = __shfl_xor_sync(0xffffffffu, x, o);
        x = w == 0 ? Op0::op(x, y) : x + y;
      }
      if (wl == 0) sh.res[w] = x;
    }
    __syncthreads();
    if (threadIdx.x == 0) fin(sh.res);
    __syncthreads();
    return true;
  }

  __device__ void publish(V* b, V v) {
    if (owner) b[row] = v;
  }

  // Returns false when a wait ran out.
  __device__ bool solve() {
    const V Z = V(0);
    V g = Z, lo = Z, hi = Z, m = V(1);
    if (owner) {
      g = V(A.gr[row]);
      lo = box_lo(A.lo[row], V());
      hi = box_hi(A.hi[row], V());
      if (A.mi) m = A.mi[row];
    }
    V s = Z, Hs = Z, t1, t2 = Z;
    int restarts = 0, hvc = 0, hvs = 0;
    if (threadIdx.x == 0) {
      sh.used = 0;
      sh.have = 0;
      sh.tol = -1.0;
    }
    // Cauchy point: exact minimiser along the movable part of -g, halved until
    // the model decreases enough on the projected path
    const bool mv = (g < Z && hi > Z) || (g > Z && lo < Z);
    t1 = mv ? g : Z;
    publish(A.b0, t1);
    if (!sums<2, OpMax>({double(t1 < Z ? -t1 : t1), double(t1 * t1)}, [&](double* r) {
          sh.state = r[0] > 0.0;
          sh.t = A.delta / r[0];
          sh.tt1 = r[1];
        }))
      return false;
    if (sh.state) {
      t2 = product(A.b0, nullptr, Z);
      ++hvc;
      if (!sums<1>({double(t1 * t2)}, [&](double* r) {
            sh.k1 = r[0];
            if (r[0] > 0.0) sh.t = fmin(sh.t, sh.tt1 / r[0]);
            sh.tt = V(sh.t);
          }))
        return false;
      for (int bt = 0; bt <= A.backtracks; ++bt) {
        const V tt = sh.tt, di = -tt * g;
        s = clamp_v(di, lo, hi);
        Hs = -tt * t2;
        publish(A.b1, s);
        auto test = [&](double a0, double a1) {
          sh.m_s = a0 + 0.5 * a1;
          sh.have = sh.m_s <= A.cauchy_c * a0;
          sh.t *= 0.5;
          sh.tt = V(sh.t);
        };
        if (!sums<1>({mv && s != di ? 1.0 : 0.0}, [&](double* r) {
              sh.state = r[0] == 0.0;
              if (sh.state) test(-double(tt) * sh.tt1, double(tt) * double(tt) * sh.k1);
            }))
          return false;
        if (!sh.state) {
          Hs = product(A.b1, nullptr, Z);
          ++hvc;
          if (!sums<2>({double(g * s), double(s * Hs)}, [&](double* r) { test(r[0], r[1]); })) return false;
        }
        if (sh.have) break;
      }
      if (!sh.have) s = Z;
    }
    while (sh.have && sh.used < A.cg_max) {
      // CG on the free set of s
      V w = Z, p = Z, r, z, ga, gb;
      {
        const V la = lo - s, lb = hi - s;
        const bool fr = la < Z && Z < lb;
        r = fr ? -(g + Hs) : Z;
        z = m * r;
        ga = fr ? la : Z;
        gb = fr ? lb : Z;
      }
      publish(A.z, z);
      if (!sums<2>({double(r * r), double(r * z)}, [&](double* e) {
            const double nr = sqrt(e[0]);
            if (sh.tol < 0.0) sh.tol = fmin(0.1, sqrt(nr)) * nr;
            sh.rz = e[1];
            sh.tol2 = sh.tol * sh.tol;
            sh.state = nr <= sh.tol || e[0] == 0.0 ? CG_CONV : CG_RUNNING;
          }))
        return false;
      bool first = true;
      V *pold = A.pa, *pnew = A.pb;
      while (sh.state == CG_RUNNING) {
        const V be = sh.beta;
        p = first ? z : fma_v(be, p, z);
        publish(pnew, p);
        const V q = first ? product(A.z, nullptr, Z) : product(pold, A.z, be);
        first = false;
        if (!sums<1>({double(p * q)}, [&](double* k) {
              ++sh.used;
              if (k[0] <= 0.0) sh.state = CG_NEGCURV;
              else sh.alpha = V(sh.rz / k[0]);
            }))
          return false;
        if (sh.state != CG_RUNNING) break;
        const V al = sh.alpha;
        w = w + al * p;
        r = r - al * (ga < Z ? q : Z);
        z = m * r;
        publish(A.z, z);
        if (!sums<3>({double(r * r), w < ga || w > gb ? 1.0 : 0.0, double(r * z)}, [&](double* u) {
              if (u[1] > 0.0) {
                sh.state = CG_LEAVE;
              } else if (u[0] <= sh.tol2) {
                sh.state = CG_CONV;
              } else if (sh.used >= A.cg_max) {
                sh.state = CG_BUDGET;
              } else {
                sh.beta = V(u[2] / sh.rz);
                sh.rz = u[2];
              }
            }))
          return false;
        V* sw = pold;
        pold = pnew;
        pnew = sw;
      }
      const int state = sh.state;
      if (state == CG_NEGCURV) {
        // to the box along p
        V am = V(INFINITY);
        if (p > Z) am = (gb - w) / p;
        if (p < Z) am = (ga - w) / p;
        if (!sums<1, OpMin>({double(am)}, [&](double* r_) { sh.amax = V(fmax(r_[0], 0.0)); })) return false;
        if (isfinite(sh.amax)) w += sh.amax * p;
      } else if (state != CG_LEAVE) {
        s += w;
        break;
      }
      // projected search along w
      V b = V(1);
      for (int bt = 0; bt <= A.backtracks; ++bt, b *= V(0.5)) {
        t1 = clamp_v(s + b * w, lo, hi);
        publish(A.b0, t1);
        if (!barrier()) return false;
        t2 = product(A.b0, nullptr, Z);
        ++hvs;
        if (!sums<3>({double(g * t1), double(t1 * t2), double((g + Hs) * (t1 - s))}, [&](double* a) {
              const double m_t = a[0] + 0.5 * a[1];
              sh.have = m_t <= sh.m_s + A.cauchy_c * a[2];
              if (sh.have) sh.m_s = m_t;
            }))
          return false;
        if (sh.have) break;
      }
      if (!sh.have) break;
      s = t1;
      Hs = t2;
      if (++restarts > A.max_restarts) break;
    }
    if (owner) A.s[row] = double(clamp_v(s, lo, hi));
    if (blockIdx.x == 0 && threadIdx.x == 0) {
      A.ctl->base = target;
      A.ctl->used = sh.used;
      A.ctl->restarts = restarts;
      A.ctl->hv_cauchy = hvc;
      A.ctl->hv_search = hvs;
    }
    return true;
  }
};

template <int D, class TS, class V, bool CACHE>
__global__ void __launch_bounds__(kThreads, 2) k_subproblem(SubArgs<D, TS, V> args) {
  __shared__ typename Sub<D, TS, V, CACHE>::Shared sh;
  Sub<D, TS, V, CACHE> S(args, sh);
  S.solve();
}

template <int D, class TS, class V, bool CACHE>
cudaError_t launch(SubArgs<D, TS, V> args, cudaStream_t st) {
  // CTAs that fit the device at once (once per device and thread)
  static thread_local int dev_of = -1, cap = 0, sms_of = 1;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev_of != dev) {
    int coop = 0, sms = 0, per = 0;
    if ((e = cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev)) != cudaSuccess) return e;
    if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_subproblem<D, TS, V, CACHE>, kThreads, 0);
    if (e != cudaSuccess) return e;
    cap = coop ? std::min(per * sms, kMaxCoopBlocks) : 0;
    sms_of = sms;
    dev_of = dev;
  }
  // rows spread over as many SMs as there are, in whole warps
  const long long n = (D + 1) * args.g.N;
  args.rows = int(std::min<long long>(kLanes, ((n + sms_of - 1) / sms_of + 31) / 32 * 32));
  const long long nb = (n + args.rows - 1) / args.rows;
  if (nb > cap) return cudaErrorNotSupported;
  void* kargs[] = {&args};
  return cudaLaunchCooperativeKernel((const void*)k_subproblem<D, TS, V, CACHE>, dim3(unsigned(nb)),
                                     dim3(kThreads), kargs, 0, st);
}

template <int D, class TS, class V>
SubArgs<D, TS, V> make_args(const Geom& g, const SubIn& in) {
  SubArgs<D, TS, V> a;
  a.g = g;
  a.S = static_cast<const TS*>(in.stencil);
  a.gr = in.gr;
  a.lo = in.lo;
  a.hi = in.hi;
  a.mi = static_cast<const V*>(in.mi);
  a.s = in.s;
  V* w = static_cast<V*>(in.work);
  const long long n = (D + 1) * g.N;
  a.b0 = w;
  a.b1 = w + n;
  a.z = w + 2 * n;
  a.pa = w + 3 * n;
  a.pb = w + 4 * n;
  a.partials = in.partials;
  a.bar = in.bar;
  a.ctl = in.ctl;
  a.delta = in.delta;
  a.cauchy_c = in.cauchy_c;
  a.spin_limit = in.spin_limit;
  a.backtracks = in.backtracks;
  a.cg_max = in.cg_max;
  a.max_restarts = in.max_restarts;
  return a;
}

}  // namespace

// At most this many rows go to the one-launch solve: those that 152 SMs hold
// with two CTAs of 128 rows each (65^2 and 113^2 nodes in 2D, 21^3 in 3D).
bool subproblem_small(const Geom& g) { return (g.dim + 1) * g.N <= 38912; }

cudaError_t subproblem_coop(const Geom& g, const SubIn& in, cudaStream_t st) {
  if (!subproblem_small(g)) return cudaErrorNotSupported;
  if (in.fp32) {
    return g.dim == 3 ? launch<3, float, float, true>(make_args<3, float, float>(g, in), st)
                      : launch<2, float, float, true>(make_args<2, float, float>(g, in), st);
  }
  return g.dim == 3 ? launch<3, double, double, false>(make_args<3, double, double>(g, in), st)
                    : launch<2, double, double, true>(make_args<2, double, double>(g, in), st);
}

}  // namespace pf
