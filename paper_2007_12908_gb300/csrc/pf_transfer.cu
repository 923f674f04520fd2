// Transfers between a coarse grid and its 2:1 refinement: Q1 interpolation
// I, restriction R = I^T, projection P = diag(R 1)^-1 R (Sec. 3) and the
// coarse feasible set (Sec. 3.2).
//
// These are streaming passes (one fine vector in or out), but on this chip
// FP64 arithmetic runs at 2 lanes per SM and clock, so a pass that spends
// more than about one FP64 instruction per fine value is bound by that pipe
// and not by memory: one thread per output value with the tensor-product
// weights formed and multiplied in FP64 took 133-149 us a pass at 129^3
// (FP64 pipe 81-88 % busy, DRAM under 10 %).  Here a thread owns one coarse
// (x, y) column of a plane and marches along z:
//  - the sums are factored axis by axis, so a fine layer's x and y sums are
//    formed once and shared by the two coarse layers it touches;
//  - an average is one addition, a/2 + b/2 with the halves taken off the
//    exponent in integer arithmetic, so prolongation needs 8 FP64 instructions
//    per 2^3 fine nodes and restriction 18 per coarse node;
//  - the bounds compare order-preserving integer keys and use no FP64
//    instruction at all;
//  - the only divisions left are P's at nodes on a face (the weight sum is a
//    power of two elsewhere); the columns on x and y faces are numbered after
//    all others, so that no warp divides for a lane or two.
// Columns are numbered along rows without gaps: an FP64 instruction takes
// its 16 cycles also for a warp with one live lane, and rows of 65 coarse
// nodes in tiles of 32 cost a half more than they need.
#include <algorithm>
#include <cmath>

#include "pf_internal.h"
#include "pf_launch.cuh"

namespace pf {

namespace {

constexpr int kThreads = 128;

// x / 2 in integer arithmetic, rounded to even where the result is subnormal
// (an FP64 multiplication would take the pipe that bounds these passes).
// The words are taken apart as 32-bit integers: a 64-bit mask of the sign is
// compiled into an FP64 instruction.
__device__ __forceinline__ double half_of(double x) {
  const int hi = __double2hiint(x), lo = __double2loint(x);
  const unsigned e = (unsigned(hi) >> 20) & 0x7ffu;
  if (e - 2u < 0x7fdu) return __hiloint2double(hi - (1 << 20), lo);
  if (e == 0x7ffu) return x;
  const unsigned m = unsigned(hi) & 0x7fffffffu;
  const unsigned ql = __funnelshift_r(unsigned(lo), m, 1), qh = m >> 1;
  const unsigned up = unsigned(lo) & ql & 1u, rl = ql + up;
  const unsigned rh = (unsigned(hi) & 0x80000000u) | (qh + (rl < ql ? 1u : 0u));
  return __hiloint2double(int(rh), int(rl));
}
__device__ __forceinline__ float half_of(float x) { return 0.5f * x; }

// (a + b) / 2 without an intermediate that can overflow; the halves of a
// value used twice are formed once
template <class T>
__device__ __forceinline__ T avg(T a, T b) {
  return half_of(a) + half_of(b);
}

__device__ __forceinline__ double add_half(double a, double b) { return __fma_rn(0.5, b, a); }
__device__ __forceinline__ float add_half(float a, float b) { return __fmaf_rn(0.5f, b, a); }

// A thread's column, plane and range of coarse layers from the block's linear
// index b (a plain 1D grid: axes of up to 2^20 nodes exceed grid.y and .z).
// Columns off the x and y faces come first, in rows, then those on them.
struct Column {
  int x, y, f, z0, z1;  // z1 exclusive
  bool live;
};
__device__ __forceinline__ Column my_column(const Geom& gc, unsigned blocks_xy, unsigned chunks,
                                            int chunk, unsigned b) {
  Column c;
  long long t = (long long)(b % blocks_xy) * kThreads + threadIdx.x;
  b /= blocks_xy;
  c.z0 = int(b % chunks) * chunk;
  c.z1 = min(c.z0 + chunk, gc.n[2]);
  c.f = int(b / chunks);
  const int n0 = gc.n[0], n1 = gc.n[1], w = n0 - 2;
  c.live = t < (long long)n0 * n1;
  const long long inner = (long long)w * (n1 - 2);
  if (t < inner) {
    if (inner <= 0xffffffffLL) {
      c.y = 1 + int(unsigned(t) / unsigned(w));
      c.x = 1 + int(unsigned(t) % unsigned(w));
    } else {
      c.y = 1 + int(t / w);
      c.x = 1 + int(t % w);
    }
  } else {
    t -= inner;
    if (t < 2LL * n0) {
      c.y = t < n0 ? 0 : n1 - 1;
      c.x = int(t < n0 ? t : t - n0);
    } else {
      t -= 2LL * n0;
      c.y = 1 + int(t >> 1);
      c.x = (t & 1) ? n0 - 1 : 0;
    }
  }
  return c;
}

// Prolongation: a fine node on an even index coincides with a coarse node,
// on an odd index it averages its two coarse neighbours, axis by axis.
// 149 -> 26 us at 129^3.
template <class T>
__global__ void __launch_bounds__(kThreads)
    k_prolong(Geom gc, Geom gf, unsigned blocks_xy, unsigned chunks, int chunk,
              const T* __restrict__ in, T* __restrict__ out, const int* skip) {
  const unsigned blk = launch_wait_block();
  if (skip && *skip) return;
  const Column c = my_column(gc, blocks_xy, chunks, chunk, blk);
  if (!c.live) return;
  const bool hx = c.x + 1 < gc.n[0], hy = c.y + 1 < gc.n[1];
  const long long cl = (long long)gc.n[0] * gc.n[1], fl = (long long)gf.n[0] * gf.n[1];
  const T* src = in + c.f * gc.N + c.x + (long long)gc.n[0] * c.y;
  T* dst = out + c.f * gf.N + 2 * c.x + (long long)gf.n[0] * (2 * c.y);
  const int dx = hx ? 1 : 0;
  const long long dy = hy ? gc.n[0] : 0, fy = hy ? gf.n[0] : 0;
  // no branches: past the last column or row the odd nodes fall on the even
  // one, which is written after them
  auto load = [&](int z, T (&v)[4]) {
    const T* s = src + z * cl;
    const T c00 = s[0], c10 = s[dx], c01 = s[dy], c11 = s[dy + dx];
    v[0] = c00;
    v[1] = avg(c00, c10);
    v[2] = avg(c00, c01);
    v[3] = avg(v[1], avg(c01, c11));
  };
  auto put = [&](long long zf, const T (&v)[4]) {
    T* d = dst + zf * fl;
    d[fy + dx] = v[3];
    d[fy] = v[2];
    d[dx] = v[1];
    d[0] = v[0];
  };
  T prev[4];
  load(c.z0, prev);
  put(2LL * c.z0, prev);
  const int last = min(c.z1, gc.n[2] - 1);
  for (int z = c.z0 + 1; z <= last; ++z) {
    T cur[4], mid[4];
    load(z, cur);
#pragma unroll
    for (int k = 0; k < 4; ++k) mid[k] = avg(prev[k], cur[k]);
    put(2LL * z - 1, mid);
    if (z < c.z1) put(2LL * z, cur);
#pragma unroll
    for (int k = 0; k < 4; ++k) prev[k] = cur[k];
  }
}

// The 3^D fine neighbourhood of a column's coarse nodes combined axis by
// axis with op(centre, neighbour); a neighbour outside the grid counts as
// op.none(centre).  The nine loads of a layer do not depend on one another
// or on a branch (addresses are clamped).  layer(z) is the x-y combination
// of fine layer z around the column.
template <class T, class Op>
struct Gather {
  const T* src;      // fine (2x, 2y, 0) of the column's plane
  long long fl;      // fine layer stride
  long long dn, up;  // offsets of rows 2y - 1 and 2y + 1 (0 outside)
  int lf, rt;        // offsets of columns 2x - 1 and 2x + 1 (0 outside)
  Op op;
  __device__ __forceinline__ T at(T centre, T v, bool inside) const {
    return inside ? op.load(v) : op.none(centre);
  }
  __device__ __forceinline__ T layer(long long z) const {
    const T* p = src + z * fl;
    T v[3][3];
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      const T* r = p + (j == 0 ? 0 : j == 1 ? dn : up);
      v[j][0] = r[0];
      v[j][1] = r[lf];
      v[j][2] = r[rt];
    }
    T row[3];
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      const T c = op.load(v[j][0]);
      row[j] = op(op(c, at(c, v[j][1], lf != 0)), at(c, v[j][2], rt != 0));
    }
    return op(op(row[0], dn != 0 ? row[1] : op.none(row[0])), up != 0 ? row[2] : op.none(row[0]));
  }
};

template <class T>
struct OpHalf {
  __device__ __forceinline__ T load(T x) const { return x; }
  __device__ __forceinline__ T none(T) const { return T(0); }
  __device__ __forceinline__ T operator()(T a, T b) const { return add_half(a, b); }
};

template <class T, class Op>
__device__ __forceinline__ Gather<T, Op> gather_of(const Column& c, const Geom& gf, const T* in,
                                                   Op op) {
  Gather<T, Op> g;
  g.fl = (long long)gf.n[0] * gf.n[1];
  g.src = in + c.f * gf.N + 2 * c.x + (long long)gf.n[0] * (2 * c.y);
  g.lf = c.x > 0 ? -1 : 0;
  g.rt = 2 * c.x + 1 < gf.n[0] ? 1 : 0;
  g.dn = c.y > 0 ? -gf.n[0] : 0;
  g.up = 2 * c.y + 1 < gf.n[1] ? gf.n[0] : 0;
  g.op = op;
  return g;
}

// Restriction R = I^T: a coarse node collects the fine nodes within one fine
// spacing, weight 1 on the coincident node and 1/2 per odd offset and axis.
// With normalise, the sum is divided by the sum of the weights (P): 8 (4 in
// 2D) inside, a factor 3/4 less per face the node lies on.
// 133 -> 52 us (R) and 58 us (P) at 129^3, FP64 pipe 79 % busy.
template <int D, class T>
__global__ void __launch_bounds__(kThreads)
    k_restrict(Geom gc, Geom gf, unsigned blocks_xy, unsigned chunks, int chunk,
               const T* __restrict__ in, T* __restrict__ out, bool normalise,
               const int* skip) {
  const unsigned blk = launch_wait_block();
  if (skip && *skip) return;
  const Column c = my_column(gc, blocks_xy, chunks, chunk, blk);
  if (!c.live) return;
  const auto g = gather_of<T, OpHalf<T>>(c, gf, in, OpHalf<T>());
  const long long cl = (long long)gc.n[0] * gc.n[1];
  T* dst = out + c.f * gc.N + c.x + (long long)gc.n[0] * c.y;
  const int faces_xy = (g.lf ? 0 : 1) + (g.rt ? 0 : 1) + (g.dn ? 0 : 1) + (g.up ? 0 : 1);
  T below = T(0);
  if (D == 3 && c.z0 > 0) below = g.layer(2LL * c.z0 - 1);
  for (int z = c.z0; z < c.z1; ++z) {
    T v = g.layer(2LL * z);
    int faces = faces_xy;
    if (D == 3) {
      if (z > 0) v = add_half(v, below);
      else ++faces;
      if (2 * z + 1 < gf.n[2]) {
        below = g.layer(2LL * z + 1);
        v = add_half(v, below);
      } else {
        ++faces;
      }
    }
    if (normalise) {
      if (faces == 0) {
        v = v * T(D == 3 ? 0.125 : 0.25);
      } else {
        T w = T(D == 3 ? 8 : 4);
        for (int k = 0; k < faces; ++k) w *= T(0.75);  // exact: 2^D (3/4)^faces
        v = v / w;
      }
    }
    dst[z * cl] = v;
  }
}

// Doubles as signed integers in the same order; a NaN lies outside the keys
// of the infinities, on the side of its sign.
__device__ __forceinline__ long long flip_key(long long b) {
  return b ^ ((b >> 63) & 0x7fffffffffffffffLL);
}
constexpr long long kKeyInf = 0x7ff0000000000000LL;      // key of +inf
constexpr long long kKeyNegInf = -0x7ff0000000000001LL;  // key of -inf

struct OpKeyMax {
  static constexpr long long start = kKeyNegInf;
  __device__ __forceinline__ long long load(long long b) const { return flip_key(b); }
  __device__ __forceinline__ long long none(long long centre) const { return centre; }
  __device__ __forceinline__ long long operator()(long long a, long long b) const { return a > b ? a : b; }
};
struct OpKeyMin {
  static constexpr long long start = kKeyInf;
  __device__ __forceinline__ long long load(long long b) const { return flip_key(b); }
  __device__ __forceinline__ long long none(long long centre) const { return centre; }
  __device__ __forceinline__ long long operator()(long long a, long long b) const { return a < b ? a : b; }
};
// The same with NaNs replaced by the start value, so that they never win (as
// with fmax / fmin): taken only where a column's result is a NaN's key.
template <class Op>
struct OpNoNan : Op {
  __device__ __forceinline__ long long load(long long b) const {
    const long long k = flip_key(b);
    return k > kKeyInf || k < kKeyNegInf ? Op::start : k;
  }
};

template <int D, class Op>
__device__ __forceinline__ void bound_column(const Column& c, const Geom& gc, const Geom& gf,
                                             const long long* in, long long* out) {
  const Op op;
  const auto g = gather_of<long long, Op>(c, gf, in, op);
  const long long cl = (long long)gc.n[0] * gc.n[1];
  long long* dst = out + c.f * gc.N + c.x + (long long)gc.n[0] * c.y;
  long long below = Op::start;
  if (D == 3 && c.z0 > 0) below = g.layer(2LL * c.z0 - 1);
  for (int z = c.z0; z < c.z1; ++z) {
    long long v = g.layer(2LL * z);
    if (D == 3) {
      v = op(v, below);
      below = Op::start;
      if (2 * z + 1 < gf.n[2]) {
        below = g.layer(2LL * z + 1);
        v = op(v, below);
      }
    }
    if (v > kKeyInf || v < kKeyNegInf) {
      const auto h = gather_of<long long, OpNoNan<Op>>(c, gf, in, OpNoNan<Op>());
      v = op(Op::start, h.layer(2LL * z));
      if (D == 3 && z > 0) v = op(v, h.layer(2LL * z - 1));
      if (D == 3 && 2 * z + 1 < gf.n[2]) v = op(v, h.layer(2LL * z + 1));
    }
    dst[z * cl] = flip_key(v);
  }
}

// Coarse feasible set: lo_c = max of lo_f, hi_c = min of hi_f over the fine
// support of each coarse basis function.  122 -> 40 us at 129^3 (two fine
// vectors).
template <int D>
__global__ void __launch_bounds__(kThreads)
    k_bounds(Geom gc, Geom gf, unsigned blocks_xy, unsigned chunks, int chunk, int nf,
             const long long* __restrict__ lo_f, const long long* __restrict__ hi_f,
             long long* __restrict__ lo_c, long long* __restrict__ hi_c) {
  const unsigned blk = launch_wait_block();
  // planes 0 .. nf-1: lo, nf .. 2 nf - 1: hi
  Column c = my_column(gc, blocks_xy, chunks, chunk, blk);
  if (!c.live) return;
  if (c.f < nf) {
    bound_column<D, OpKeyMax>(c, gc, gf, lo_f, lo_c);
  } else {
    c.f -= nf;
    bound_column<D, OpKeyMin>(c, gc, gf, hi_f, hi_c);
  }
}

// Launch shape: blocks of columns x chunks of coarse layers x planes.  A
// chunk re-reads one fine layer (or one coarse layer) of its neighbour, so
// chunks are as long as four layers (5 % more work than eight, but twice the
// blocks to even out between the SMs) where that still gives eight blocks
// per SM.
struct Shape {
  unsigned blocks_xy, chunks, blocks;
  int chunk;
  bool ok;
};
Shape shape_of(const Geom& gc, int planes) {
  Shape s;
  const long long bxy = ((long long)gc.n[0] * gc.n[1] + kThreads - 1) / kThreads;
  long long blocks = 0;
  for (s.chunk = 4;; s.chunk /= 2) {
    s.chunks = unsigned((gc.n[2] + s.chunk - 1) / s.chunk);
    blocks = bxy * s.chunks * planes;
    if (s.chunk == 1 || blocks >= 8 * 152) break;
  }
  s.ok = blocks <= 0x7fffffffLL;
  s.blocks_xy = unsigned(bxy);
  s.blocks = unsigned(blocks);
  return s;
}

template <class T>
cudaError_t prolong_t(const Geom& gc, const Geom& gf, int nf, const void* in, void* out,
                      cudaStream_t st, const int* skip) {
  const Shape s = shape_of(gc, nf);
  if (!s.ok) return cudaErrorInvalidConfiguration;
  const T* i = static_cast<const T*>(in);
  T* o = static_cast<T*>(out);
  launch_dependent(k_prolong<T>, dim3(s.blocks), dim3(kThreads), st, gc, gf, s.blocks_xy, s.chunks, s.chunk,
                   i, o, skip);
  return cudaGetLastError();
}

template <class T>
cudaError_t restrict_t(const Geom& gc, const Geom& gf, int nf, const void* in, void* out,
                       bool normalise, cudaStream_t st, const int* skip) {
  const Shape s = shape_of(gc, nf);
  if (!s.ok) return cudaErrorInvalidConfiguration;
  const T* i = static_cast<const T*>(in);
  T* o = static_cast<T*>(out);
  if (gc.dim == 3)
    launch_dependent(k_restrict<3, T>, dim3(s.blocks), dim3(kThreads), st, gc, gf, s.blocks_xy, s.chunks,
                     s.chunk, i, o, normalise, skip);
  else
    launch_dependent(k_restrict<2, T>, dim3(s.blocks), dim3(kThreads), st, gc, gf, s.blocks_xy, s.chunks,
                     s.chunk, i, o, normalise, skip);
  return cudaGetLastError();
}

}  // namespace

cudaError_t xfer_prolong(const Geom& gc, const Geom& gf, int nf, const void* in, void* out,
                         int prec, cudaStream_t st, const int* skip) {
  return prec ? prolong_t<float>(gc, gf, nf, in, out, st, skip)
              : prolong_t<double>(gc, gf, nf, in, out, st, skip);
}

cudaError_t xfer_restrict(const Geom& gc, const Geom& gf, int nf, const void* in, void* out,
                          int prec, bool normalise, cudaStream_t st, const int* skip) {
  return prec ? restrict_t<float>(gc, gf, nf, in, out, normalise, st, skip)
              : restrict_t<double>(gc, gf, nf, in, out, normalise, st, skip);
}

cudaError_t xfer_bounds(const Geom& gc, const Geom& gf, int nf, const double* lo_f,
                        const double* hi_f, double* lo_c, double* hi_c, cudaStream_t st) {
  const Shape s = shape_of(gc, 2 * nf);
  if (!s.ok) return cudaErrorInvalidConfiguration;
  const auto* lf = reinterpret_cast<const long long*>(lo_f);
  const auto* hf = reinterpret_cast<const long long*>(hi_f);
  auto* lc = reinterpret_cast<long long*>(lo_c);
  auto* hc = reinterpret_cast<long long*>(hi_c);
  if (gc.dim == 3)
    launch_dependent(k_bounds<3>, dim3(s.blocks), dim3(kThreads), st, gc, gf, s.blocks_xy, s.chunks,
                     s.chunk, nf, lf, hf, lc, hc);
  else
    launch_dependent(k_bounds<2>, dim3(s.blocks), dim3(kThreads), st, gc, gf, s.blocks_xy, s.chunks,
                     s.chunk, nf, lf, hf, lc, hc);
  return cudaGetLastError();
}

}  // namespace pf
