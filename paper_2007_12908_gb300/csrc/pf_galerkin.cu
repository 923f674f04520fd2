// Stored Galerkin coarse operators (the second-order coherent level model of
// eq. (second_order_consistency) and eq. (delta_terms) under Hessian
// lagging, Sec. 4.2.1): the model Hessian of a coarse level l is
// G^l = R G^{l+1} I with G^{L-1} = H(x_lag) on the finest level.  Instead
// of applying that chain matrix-free (a finest-level product per coarse
// product), the operators are assembled once per lag into FP32 block
// stencils, 3^d points per node.
//
// With Q1 functions nested (coarse ones lie in the fine space, so I maps them
// exactly), the element matrix of a coarse element is the integral of the
// fine Gauss-point Hessian density (A, M, B at x_lag) against products of the
// coarse 1D functions.  Such a product is N_a N_b, N_a or 1 along each axis,
// and all of them are sums of the NN moments
//   mom[k][c_x, c_y, c_z] = sum over the fine Gauss points of coefficient k
//                           times NN_cx(x) NN_cy(y) NN_cz(z),
//   NN_0 = N_0^2, NN_1 = N_0 N_1, NN_2 = N_1^2 on the coarse element
// (27 x 8 floats per element in 3D, 9 x 5 in 2D), with positive weights only.
// So:
//  1. next-to-finest level: the moments from the 4^d fine Gauss points of an
//     element's children, axis by axis;
//  2. coarser levels: the moments of a parent are its children's, with
//     N'_0 = N_0 + N_1 / 2, N'_1 = N_1 / 2 (or mirrored) per axis: exact
//     re-expansion, axis by axis;
//  3. each level's stencil from the moments (pf_assemble.cu).
// A fixed order everywhere, no atomics.  Forming and storing 32 x 32 element
// matrices instead took 1,389 us (1.24 G warp instructions: 64 Gauss points
// per entry) + 177 us (I^T K I) + 148 us (490 MB of matrix rows gathered
// entry by entry) for 65^3 -> 33^3 -> 17^3; the three steps now take
// 19 + 12 + 88 us.
#include <algorithm>
#include <string>

#include "../../include/pf.h"
#include "pf_element.cuh"
#include "pf_internal.h"
#include "pf_launch.cuh"
#include "pf_stencil.cuh"

namespace pf {

namespace {

template <int D>
struct GalDims {
  static constexpr int NC = 1 << D, F = D + 1, NCF = NCoef<D>::value;
  static constexpr int W = D == 3 ? 27 : 9;     // moments per coefficient
  static constexpr int NP = D == 3 ? 64 : 16;   // fine Gauss points per coarse element
  static constexpr int EL = 32;                 // coarse elements per CTA
  static constexpr int THREADS = EL << D;       // one per child
  static constexpr size_t smem = sizeof(float) * NCF * NP * EL;
};

template <int D>
__device__ __forceinline__ long long node_index(const Geom& g, int ix, int iy, int iz) {
  return D == 3 ? ix + (long long)g.n[0] * (iy + (long long)g.n[1] * iz) : ix + (long long)g.n[0] * iy;
}

template <int D>
__device__ __forceinline__ void elem_xyz(const Geom& g, long long e, int& ex, int& ey, int& ez) {
  ex = int(e % g.ne[0]);
  const long long r = e / g.ne[0];
  ey = D == 3 ? int(r % g.ne[1]) : int(r);
  ez = D == 3 ? int(r / g.ne[1]) : 0;
}

// NN_0, NN_1, NN_2 of a coarse element at its j-th fine Gauss point along an
// axis, t = (child + xi) / 2.
__device__ __forceinline__ constexpr float gal_nn(int j, int c) {
  const double t = 0.5 * ((j >> 1) + ((j & 1) ? PF_XI1 : PF_XI0));
  return float(c == 0 ? (1 - t) * (1 - t) : (c == 1 ? t * (1 - t) : t * t));
}

// 1. Moments of the next-to-finest level gc from the finest lag (FP32 x on
// the finest grid gf).  A CTA takes 32 consecutive coarse elements: thread =
// child, whose Gauss-point coefficients go to shared memory; then warp =
// coefficient, lane = element.  Bound by FP32 issue (about 600 operations per
// child and 450 per element and coefficient).
template <int D>
__global__ void __launch_bounds__(GalDims<D>::THREADS)
    k_gal_fine(Geom gc, Geom gf, Mat<float> m, const float* __restrict__ x,
               float* __restrict__ mom) {
  using G = GalDims<D>;
  constexpr int NC = G::NC, F = G::F, EL = G::EL;
  extern __shared__ float cf_s[];  // [coefficient][point][element]
  const long long e0 = launch_wait_block() * (long long)EL;
  {
    // thread -> element and child, neighbouring threads along x
    const int cx = threadIdx.x & 1, el = (threadIdx.x >> 1) % EL, cyz = threadIdx.x / (2 * EL);
    const long long e = e0 + el;
    if (e < gc.NE) {
      int ex, ey, ez;
      elem_xyz<D>(gc, e, ex, ey, ez);
      const int cy = cyz & 1, cz = D == 3 ? cyz >> 1 : 0;
      const int fx = 2 * ex + cx, fy = 2 * ey + cy, fz = D == 3 ? 2 * ez + cz : 0;
      float xe[F][NC];
#pragma unroll
      for (int a = 0; a < NC; ++a) {
        const long long idx = node_index<D>(gf, fx + (a & 1), fy + ((a >> 1) & 1),
                                            D == 3 ? fz + ((a >> 2) & 1) : 0);
#pragma unroll
        for (int f = 0; f < F; ++f) xe[f][a] = x[f * gf.N + idx];
      }
      float cf[NC][G::NCF];
      hess_coef<D, float>(xe, m, cf);
#pragma unroll
      for (int q = 0; q < NC; ++q) {
        const int pt = (2 * cx + (q & 1)) + 4 * (2 * cy + ((q >> 1) & 1)) +
                       (D == 3 ? 16 * (2 * cz + ((q >> 2) & 1)) : 0);
#pragma unroll
        for (int k = 0; k < G::NCF; ++k) cf_s[(k * G::NP + pt) * EL + el] = cf[q][k];
      }
    }
  }
  __syncthreads();
  const int lane = threadIdx.x & 31;
  const long long e = e0 + lane;
  if (e >= gc.NE) return;
  for (int k = threadIdx.x >> 5; k < G::NCF; k += G::THREADS / 32) {
    const float* s = cf_s + k * G::NP * EL + lane;
    float acc[G::W];
#pragma unroll
    for (int w = 0; w < G::W; ++w) acc[w] = 0.f;
#pragma unroll
    for (int jz = 0; jz < (D == 3 ? 4 : 1); ++jz) {
      float t[3][3];  // [c_x][c_y]
#pragma unroll
      for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) t[i][j] = 0.f;
#pragma unroll
      for (int jy = 0; jy < 4; ++jy) {
        float r[3] = {0.f, 0.f, 0.f};
#pragma unroll
        for (int jx = 0; jx < 4; ++jx) {
          const float val = s[(jx + 4 * jy + 16 * jz) * EL];
#pragma unroll
          for (int i = 0; i < 3; ++i) r[i] = fmaf(gal_nn(jx, i), val, r[i]);
        }
#pragma unroll
        for (int i = 0; i < 3; ++i)
#pragma unroll
          for (int j = 0; j < 3; ++j) t[i][j] = fmaf(gal_nn(jy, j), r[i], t[i][j]);
      }
#pragma unroll
      for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) {
          if constexpr (D == 3) {
#pragma unroll
            for (int l = 0; l < 3; ++l)
              acc[i * 9 + j * 3 + l] = fmaf(gal_nn(jz, l), t[i][j], acc[i * 9 + j * 3 + l]);
          } else {
            acc[i * 3 + j] = t[i][j];
          }
        }
    }
#pragma unroll
    for (int w = 0; w < G::W; ++w) mom[((long long)k * G::W + w) * gc.NE + e] = acc[w];
  }
}

// A child's NN moments along one axis (c = 0 or 1: its half of the parent)
// as its part of the parent's.
__device__ __forceinline__ void to_parent(int c, const float (&w)[3], float (&o)[3]) {
  const float lo = c ? w[0] : w[2], hi = c ? w[2] : w[0];
  const float q = 0.25f * lo, h = fmaf(0.5f, w[1], q), full = (q + w[1]) + hi;
  o[0] = c ? q : full;
  o[1] = h;
  o[2] = c ? full : q;
}

// 2. Moments of the coarse level gc from those of the level above it (gf).
// One thread per (coarse element, coefficient).
template <int D>
__global__ void __launch_bounds__(128) k_gal_coarsen(Geom gc, Geom gf, const float* __restrict__ mf,
                                                     float* __restrict__ mc) {
  const unsigned blk = launch_wait_block();
  using G = GalDims<D>;
  constexpr int NL = D == 3 ? 3 : 1;
  const long long total = gc.NE * G::NCF;
  for (long long t = blk * (long long)blockDim.x + threadIdx.x; t < total;
       t += (long long)gridDim.x * blockDim.x) {
    const int k = int(t / gc.NE);
    const long long e = t - k * gc.NE;
    int ex, ey, ez;
    elem_xyz<D>(gc, e, ex, ey, ez);
    const float* src = mf + (long long)k * G::W * gf.NE;
    float acc[3][3][NL];
#pragma unroll
    for (int w = 0; w < G::W; ++w) (&acc[0][0][0])[w] = 0.f;
#pragma unroll 1
    for (int cz = 0; cz < (D == 3 ? 2 : 1); ++cz) {
      float zs[3][3][NL];  // x and y of the parent, z of the child
#pragma unroll
      for (int w = 0; w < G::W; ++w) (&zs[0][0][0])[w] = 0.f;
#pragma unroll 1
      for (int cy = 0; cy < 2; ++cy) {
        float ys[3][3][NL];  // x of the parent, y and z of the child
#pragma unroll
        for (int w = 0; w < G::W; ++w) (&ys[0][0][0])[w] = 0.f;
#pragma unroll
        for (int cx = 0; cx < 2; ++cx) {
          const long long ef = D == 3 ? (2 * ex + cx) + (long long)gf.ne[0] * ((2 * ey + cy) + (long long)gf.ne[1] * (2 * ez + cz))
                                      : (2 * ex + cx) + (long long)gf.ne[0] * (2 * ey + cy);
          const float* s = src + ef;
#pragma unroll
          for (int j = 0; j < 3; ++j)
#pragma unroll
            for (int l = 0; l < NL; ++l) {
              float w[3], o[3];
#pragma unroll
              for (int i = 0; i < 3; ++i) w[i] = s[(long long)((i * 3 + j) * NL + l) * gf.NE];
              to_parent(cx, w, o);
#pragma unroll
              for (int i = 0; i < 3; ++i) ys[i][j][l] += o[i];
            }
        }
#pragma unroll
        for (int i = 0; i < 3; ++i)
#pragma unroll
          for (int l = 0; l < NL; ++l) {
            const float w[3] = {ys[i][0][l], ys[i][1][l], ys[i][2][l]};
            float o[3];
            to_parent(cy, w, o);
#pragma unroll
            for (int j = 0; j < 3; ++j) zs[i][j][l] += o[j];
          }
      }
#pragma unroll
      for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) {
          if constexpr (D == 3) {
            const float w[3] = {zs[i][j][0], zs[i][j][1], zs[i][j][2]};
            float o[3];
            to_parent(cz, w, o);
#pragma unroll
            for (int l = 0; l < 3; ++l) acc[i][j][l] += o[l];
          } else {
            acc[i][j][0] = zs[i][j][0];
          }
        }
    }
#pragma unroll
    for (int w = 0; w < G::W; ++w) mc[((long long)k * G::W + w) * gc.NE + e] = (&acc[0][0][0])[w];
  }
}

template <class T>
Mat<T> to_mat(const Mat<double>& m) {
  Mat<T> r;
  r.lam = T(m.lam); r.mu = T(m.mu); r.Gc = T(m.Gc); r.ls = T(m.ls); r.k = T(m.k);
  r.p = T(m.p); r.inv_h = T(m.inv_h); r.w = T(m.w); r.gcl = T(m.gcl);
  r.lmu = T(m.lmu); r.hmu = T(m.hmu);
  return r;
}

int blocks_for(long long n, int threads, long long cap) {
  return int(std::max<long long>(1, std::min<long long>((n + threads - 1) / threads, cap)));
}

}  // namespace

long long galerkin_elem_count(const Geom& g) {
  return g.NE * (g.dim == 3 ? GalDims<3>::W * GalDims<3>::NCF : GalDims<2>::W * GalDims<2>::NCF);
}

long long galerkin_stencil_count(const Geom& g) {
  const int f = g.dim + 1;
  return (g.dim == 3 ? 27LL : 9LL) * f * f * g.N;
}

template <int D>
static cudaError_t launch_gal_fine(const Geom& gc, const Geom& gf, const Mat<float>& m,
                                   const float* x, float* mom, cudaStream_t st) {
  using G = GalDims<D>;
  cudaError_t e = cudaFuncSetAttribute(k_gal_fine<D>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       int(G::smem));
  if (e != cudaSuccess) return e;
  const long long nb = (gc.NE + G::EL - 1) / G::EL;
  launch_dependent(k_gal_fine<D>, dim3(unsigned(nb)), dim3(G::THREADS), size_t(G::smem), st, gc, gf, m, x, mom);
  return cudaGetLastError();
}

cudaError_t galerkin_fine(const Geom& gc, const Geom& gf, const Mat<double>& mf, const float* x_fine,
                          float* mom, cudaStream_t st) {
  return gc.dim == 3 ? launch_gal_fine<3>(gc, gf, to_mat<float>(mf), x_fine, mom, st)
                     : launch_gal_fine<2>(gc, gf, to_mat<float>(mf), x_fine, mom, st);
}

cudaError_t galerkin_coarsen(const Geom& gc, const Geom& gf, const float* mom_f, float* mom_c,
                             cudaStream_t st) {
  const int ncf = gc.dim == 3 ? GalDims<3>::NCF : GalDims<2>::NCF;
  const int nb = blocks_for(gc.NE * ncf, 128, 32LL * 1216);
  if (gc.dim == 3) launch_dependent(k_gal_coarsen<3>, dim3(nb), dim3(128), st, gc, gf, mom_f, mom_c);
  else launch_dependent(k_gal_coarsen<2>, dim3(nb), dim3(128), st, gc, gf, mom_f, mom_c);
  return cudaGetLastError();
}

cudaError_t galerkin_apply(const Geom& g, const float* S, const void* v, void* y, int prec,
                           cudaStream_t st, const int* skip) {
  if (prec == PF_FP32) {
    const float* x = static_cast<const float*>(v);
    float* o = static_cast<float*>(y);
    return g.dim == 3 ? stencil_rows<3>(g, S, x, o, st, skip) : stencil_rows<2>(g, S, x, o, st, skip);
  }
  const double* x = static_cast<const double*>(v);
  double* o = static_cast<double*>(y);
  return g.dim == 3 ? stencil_rows<3>(g, S, x, o, st, skip) : stencil_rows<2>(g, S, x, o, st, skip);
}

}  // namespace pf
