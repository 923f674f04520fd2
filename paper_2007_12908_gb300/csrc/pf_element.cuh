// Q1 element algebra of the pressurised AT2 functional (Sec. 2, eq.
// pressurized with the +p g(c) div u sign reading), evaluated per element at
// the 2^d Gauss points of a uniform cell.
//
// Interpolation to the Gauss points and the test-function contraction back to
// the corners are sum-factorised along the axes: one pass per axis, each a
// 2-point linear blend (values) or a difference (derivatives, constant along
// their own axis for Q1).  Corner a = ax + 2 ay + 4 az, Gauss point
// q = qx + 2 qy + 4 qz; 1D shape values at the Gauss points are
// N(q=0) = (XI1, XI0), N(q=1) = (XI0, XI1) with XI0 + XI1 = 1.
// Derivatives here are raw nodal differences; callers scale by 1/h.
#pragma once
#include <cuda_runtime.h>

namespace pf {

// (1 -+ 1/sqrt(3)) / 2
#define PF_XI0 0.21132486540518711775
#define PF_XI1 0.78867513459481288225

template <class T>
struct Mat {
  T lam, mu, Gc, ls, k, p;  // Lame, toughness, length scale, residual, pressure
  T inv_h;                  // 1/h
  T w;                      // Gauss weight times det J = h^d / 2^d
  T gcl;                    // Gc / ls
  T lmu, hmu;               // lam / mu, h / mu
};

// ---------------------------------------------------------------- 3D passes
template <class T>
__device__ __forceinline__ void interp3(const T f[8], T val[8], T gx[8], T gy[8], T gz[8]) {
  const T x0 = T(PF_XI0), x1 = T(PF_XI1);
  T X[2][2][2], DX[2][2];
#pragma unroll
  for (int az = 0; az < 2; ++az)
#pragma unroll
    for (int ay = 0; ay < 2; ++ay) {
      const T v0 = f[2 * ay + 4 * az], d = f[1 + 2 * ay + 4 * az] - v0;
      DX[ay][az] = d;
      X[0][ay][az] = v0 + x0 * d;
      X[1][ay][az] = v0 + x1 * d;
    }
  T XY[2][2][2], DY[2][2], DXY[2][2];
#pragma unroll
  for (int az = 0; az < 2; ++az) {
#pragma unroll
    for (int qx = 0; qx < 2; ++qx) {
      const T v0 = X[qx][0][az], d = X[qx][1][az] - v0;
      DY[qx][az] = d;
      XY[qx][0][az] = v0 + x0 * d;
      XY[qx][1][az] = v0 + x1 * d;
    }
    const T v0 = DX[0][az], d = DX[1][az] - v0;
    DXY[0][az] = v0 + x0 * d;
    DXY[1][az] = v0 + x1 * d;
  }
#pragma unroll
  for (int qy = 0; qy < 2; ++qy)
#pragma unroll
    for (int qx = 0; qx < 2; ++qx) {
      const int q = qx + 2 * qy;
      const T v0 = XY[qx][qy][0], d = XY[qx][qy][1] - v0;
      val[q] = v0 + x0 * d;
      val[q + 4] = v0 + x1 * d;
      gz[q] = d;
      gz[q + 4] = d;
    }
#pragma unroll
  for (int qy = 0; qy < 2; ++qy) {
    const T v0 = DXY[qy][0], d = DXY[qy][1] - v0;
    const T a = v0 + x0 * d, b = v0 + x1 * d;
    gx[2 * qy] = a; gx[1 + 2 * qy] = a;
    gx[2 * qy + 4] = b; gx[1 + 2 * qy + 4] = b;
  }
#pragma unroll
  for (int qx = 0; qx < 2; ++qx) {
    const T v0 = DY[qx][0], d = DY[qx][1] - v0;
    const T a = v0 + x0 * d, b = v0 + x1 * d;
    gy[qx] = a; gy[qx + 2] = a;
    gy[qx + 4] = b; gy[qx + 6] = b;
  }
}

// r[a] = sum_q s0[q] N_a(q) + sx[q] Dx_a(q) + sy[q] Dy_a(q) + sz[q] Dz_a(q)
// (raw derivatives), the adjoint of interp3.  s0 == nullptr drops the value
// term (IEEE arithmetic cannot fold multiplications by a zero term away).
template <class T>
__device__ __forceinline__ void test3(const T* s0, const T sx[8], const T sy[8], const T sz[8],
                                      T r[8]) {
  const T x0 = T(PF_XI0), x1 = T(PF_XI1);
  T XYb[2][2][2], DXYb[2][2], DYb[2][2];
#pragma unroll
  for (int qy = 0; qy < 2; ++qy)
#pragma unroll
    for (int qx = 0; qx < 2; ++qx) {
      const int q = qx + 2 * qy;
      const T zs = sz[q] + sz[q + 4];
      if (s0) {
        XYb[qx][qy][0] = x1 * s0[q] + x0 * s0[q + 4] - zs;
        XYb[qx][qy][1] = x0 * s0[q] + x1 * s0[q + 4] + zs;
      } else {
        XYb[qx][qy][0] = -zs;
        XYb[qx][qy][1] = zs;
      }
    }
#pragma unroll
  for (int qy = 0; qy < 2; ++qy) {
    const T a = sx[2 * qy] + sx[1 + 2 * qy], b = sx[2 * qy + 4] + sx[1 + 2 * qy + 4];
    DXYb[qy][0] = x1 * a + x0 * b;
    DXYb[qy][1] = x0 * a + x1 * b;
  }
#pragma unroll
  for (int qx = 0; qx < 2; ++qx) {
    const T a = sy[qx] + sy[qx + 2], b = sy[qx + 4] + sy[qx + 6];
    DYb[qx][0] = x1 * a + x0 * b;
    DYb[qx][1] = x0 * a + x1 * b;
  }
  T Xb[2][2][2], DXb[2][2];
#pragma unroll
  for (int az = 0; az < 2; ++az) {
#pragma unroll
    for (int qx = 0; qx < 2; ++qx) {
      Xb[qx][0][az] = x1 * XYb[qx][0][az] + x0 * XYb[qx][1][az] - DYb[qx][az];
      Xb[qx][1][az] = x0 * XYb[qx][0][az] + x1 * XYb[qx][1][az] + DYb[qx][az];
    }
    DXb[0][az] = x1 * DXYb[0][az] + x0 * DXYb[1][az];
    DXb[1][az] = x0 * DXYb[0][az] + x1 * DXYb[1][az];
  }
#pragma unroll
  for (int az = 0; az < 2; ++az)
#pragma unroll
    for (int ay = 0; ay < 2; ++ay) {
      r[2 * ay + 4 * az] = x1 * Xb[0][ay][az] + x0 * Xb[1][ay][az] - DXb[ay][az];
      r[1 + 2 * ay + 4 * az] = x0 * Xb[0][ay][az] + x1 * Xb[1][ay][az] + DXb[ay][az];
    }
}

// ---------------------------------------------------------------- 2D passes
template <class T>
__device__ __forceinline__ void interp2(const T f[4], T val[4], T gx[4], T gy[4]) {
  const T x0 = T(PF_XI0), x1 = T(PF_XI1);
  T X[2][2], DX[2];
#pragma unroll
  for (int ay = 0; ay < 2; ++ay) {
    const T v0 = f[2 * ay], d = f[1 + 2 * ay] - v0;
    DX[ay] = d;
    X[0][ay] = v0 + x0 * d;
    X[1][ay] = v0 + x1 * d;
  }
#pragma unroll
  for (int qx = 0; qx < 2; ++qx) {
    const T v0 = X[qx][0], d = X[qx][1] - v0;
    val[qx] = v0 + x0 * d;
    val[qx + 2] = v0 + x1 * d;
    gy[qx] = d;
    gy[qx + 2] = d;
  }
  const T v0 = DX[0], d = DX[1] - v0;
  const T a = v0 + x0 * d, b = v0 + x1 * d;
  gx[0] = a; gx[1] = a; gx[2] = b; gx[3] = b;
}

template <class T>
__device__ __forceinline__ void test2(const T* s0, const T sx[4], const T sy[4], T r[4]) {
  const T x0 = T(PF_XI0), x1 = T(PF_XI1);
  T Xb[2][2];
#pragma unroll
  for (int qx = 0; qx < 2; ++qx) {
    const T ys = sy[qx] + sy[qx + 2];
    if (s0) {
      Xb[qx][0] = x1 * s0[qx] + x0 * s0[qx + 2] - ys;
      Xb[qx][1] = x0 * s0[qx] + x1 * s0[qx + 2] + ys;
    } else {
      Xb[qx][0] = -ys;
      Xb[qx][1] = ys;
    }
  }
  const T a = sx[0] + sx[1], b = sx[2] + sx[3];
  const T DXb0 = x1 * a + x0 * b, DXb1 = x0 * a + x1 * b;
#pragma unroll
  for (int ay = 0; ay < 2; ++ay) {
    const T dxb = ay ? DXb1 : DXb0;
    r[2 * ay] = x1 * Xb[0][ay] + x0 * Xb[1][ay] - dxb;
    r[1 + 2 * ay] = x0 * Xb[0][ay] + x1 * Xb[1][ay] + dxb;
  }
}

// ---------------------------------------------------------------- dispatch
template <int D, class T>
__device__ __forceinline__ void interp(const T* f, T* val, T (*g)[1 << D]) {
  if constexpr (D == 3) interp3<T>(f, val, g[0], g[1], g[2]);
  else interp2<T>(f, val, g[0], g[1]);
}

template <int D, class T>
__device__ __forceinline__ void test(const T* s0, T (*s1)[1 << D], T* r) {
  if constexpr (D == 3) test3<T>(s0, s1[0], s1[1], s1[2], r);
  else test2<T>(s0, s1[0], s1[1], r);
}

template <int D, class T>
__device__ __forceinline__ void zero_test(T* r) {
#pragma unroll
  for (int a = 0; a < (1 << D); ++a) r[a] = T(0);
}

// Strain of a displacement gradient G[i][k] = d u_i / d x_k.
template <int D, class T>
struct Strain {
  T eps[D][D];
  T tr;
  __device__ __forceinline__ void set(const T G[D][D]) {
    tr = T(0);
#pragma unroll
    for (int i = 0; i < D; ++i) {
      tr += G[i][i];
#pragma unroll
      for (int k = 0; k < D; ++k) eps[i][k] = T(0.5) * (G[i][k] + G[k][i]);
    }
  }
  __device__ __forceinline__ T ddot(const Strain& o) const {
    T s = T(0);
#pragma unroll
    for (int i = 0; i < D; ++i)
#pragma unroll
      for (int k = 0; k < D; ++k) s += eps[i][k] * o.eps[i][k];
    return s;
  }
};

template <int D>
struct NSym {
  static constexpr int value = D * (D + 1) / 2;  // B stored 00, 11, (22), 01, (02, 12)
};
template <int D>
struct NCoef {
  static constexpr int value = NSym<D>::value + 2;  // A, M, B
};

template <int D>
__device__ __forceinline__ constexpr int sym_index(int i, int k) {
  if (i == k) return i;
  if (D == 2) return 2;
  const int lo = i < k ? i : k, hi = i < k ? k : i;
  return lo == 0 ? (hi == 1 ? 3 : 4) : 5;
}

// ---------------------------------------------------------------- element ops
// Every op takes the element's nodal values xe[f][a] (f = field plane,
// a = corner) and, for hessvec / energy_diff, a second vector ve[f][a].

// ---------------------------------------------------------------- Gauss values
// Values and derivatives at the Gauss points from differences of corner values,
// taken before anything is interpolated (a translation of the field does not
// enter them), each point from its nearest corner: XI0 (0.21) is the weight of
// every difference and of its rounding.  As monomials in coordinates from one
// corner (weights up to XI1 = 0.79, errors of the far points in common) the
// energy and the gradient of a rough element had 1.4 to 1.6 times this rounding,
// for less arithmetic: FP64 operators on 65 x 49 x 57 3,214 us, now 3,245, double-float
// energy and gradient of 97 x 105 x 89 nodes 557, now 596, the batched 2D case
// 1,167, now 1,229.  A mixed difference serves both of its axes.
// FP64 and double-float instructions are what bounds energy, gradient and
// Hessian coefficients (in 3D 2 lanes of FP64 per SM and clock; some 13
// instructions per double-float operation).

// a b + c
template <class T>
__device__ __forceinline__ T madd(T a, T b, T c) { return a * b + c; }
// 2 x
template <class T>
__device__ __forceinline__ T twice(T x) { return x + x; }

// the two Gauss points between p and q
template <class T>
__device__ __forceinline__ void lerp(T p, T q, T& o0, T& o1) {
  const T d = q - p;
  o0 = madd(T(PF_XI0), d, p);
  o1 = madd(T(-PF_XI0), d, q);
}

// KEEP holds the differences along z, which are otherwise formed again in each
// layer of Gauss points (8 values of a field in registers instead of 16).
template <class T, bool KEEP>
struct Corners3 {
  T f[8], z[4], xz[2], yz[2];  // z by corner, mixed differences by ay and ax
  __device__ __forceinline__ void set(const T g[8]) {
#pragma unroll
    for (int k = 0; k < 8; ++k) f[k] = g[k];
    differences(f, f + 4, z, xz, yz);
  }
  // z-derivative at Gauss point (qx, qy), independent of z
  __device__ __forceinline__ void dz(T (&o)[2][2]) const {
    const T t = T(PF_XI0);
    lerp(madd(t, xz[0], z[0]), madd(t, xz[1], z[2]), o[0][0], o[0][1]);
    lerp(madd(-t, xz[0], z[1]), madd(-t, xz[1], z[3]), o[1][0], o[1][1]);
  }
  // in Gauss layer qz: x-derivative by qy, y-derivative by qx
  __device__ __forceinline__ void dxy(int qz, T (&gx)[2], T (&gy)[2]) const {
    T n[4], d[4], dxz[2], dyz[2];
    const T t = T(PF_XI0), tz = layer(qz, n, d, dxz, dyz);
    // x-derivative by ay and y-derivative by ax at the layer's height
    const T a0 = madd(tz, dxz[0], n[1] - n[0]), a1 = madd(tz, dxz[1], n[3] - n[2]);
    const T b0 = madd(tz, dyz[0], n[2] - n[0]), b1 = madd(tz, dyz[1], n[3] - n[1]);
    const T m = a1 - a0;
    gx[0] = madd(t, m, a0);
    gx[1] = madd(-t, m, a1);
    gy[0] = madd(t, m, b0);
    gy[1] = madd(-t, m, b1);
  }
  // the values v[qx][qy] of the layer
  __device__ __forceinline__ void values(int qz, T (&v)[2][2]) const {
    T n[4], d[4], dxz[2], dyz[2], e[2][2];  // e[qx][ay]
    const T tz = layer(qz, n, d, dxz, dyz);
#pragma unroll
    for (int ay = 0; ay < 2; ++ay)
      lerp(madd(tz, d[2 * ay], n[2 * ay]), madd(tz, d[2 * ay + 1], n[2 * ay + 1]), e[0][ay], e[1][ay]);
#pragma unroll
    for (int qx = 0; qx < 2; ++qx) lerp(e[qx][0], e[qx][1], v[qx][0], v[qx][1]);
  }

 private:
  static __device__ __forceinline__ void differences(const T* n, const T* m, T (&d)[4], T (&dxz)[2], T (&dyz)[2]) {
#pragma unroll
    for (int k = 0; k < 4; ++k) d[k] = m[k] - n[k];
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      dxz[k] = d[2 * k + 1] - d[2 * k];
      dyz[k] = d[k + 2] - d[k];
    }
  }
  // the layer's nearer corners n, the differences and their weight
  __device__ __forceinline__ T layer(int qz, T (&n)[4], T (&d)[4], T (&dxz)[2], T (&dyz)[2]) const {
#pragma unroll
    for (int k = 0; k < 4; ++k) n[k] = qz ? f[k + 4] : f[k];
    if constexpr (KEEP) {
#pragma unroll
      for (int k = 0; k < 4; ++k) d[k] = z[k];
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        dxz[k] = xz[k];
        dyz[k] = yz[k];
      }
      return qz ? T(-PF_XI0) : T(PF_XI0);
    } else {
      T m[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) m[k] = qz ? f[k] : f[k + 4];
      differences(n, m, d, dxz, dyz);
      return T(PF_XI0);
    }
  }
};

template <class T>
struct Corners2 {
  T f[4], x[2], y[2], xy;
  __device__ __forceinline__ void set(const T g[4]) {
#pragma unroll
    for (int k = 0; k < 4; ++k) f[k] = g[k];
    x[0] = f[1] - f[0];
    x[1] = f[3] - f[2];
    y[0] = f[2] - f[0];
    y[1] = f[3] - f[1];
    xy = x[1] - x[0];
  }
  __device__ __forceinline__ void dxy(T (&gx)[2], T (&gy)[2]) const {
    const T t = T(PF_XI0);
    gx[0] = madd(t, xy, x[0]);
    gx[1] = madd(-t, xy, x[1]);
    gy[0] = madd(t, xy, y[0]);
    gy[1] = madd(-t, xy, y[1]);
  }
  __device__ __forceinline__ void values(T (&v)[2][2]) const {
    const T t = T(PF_XI0);
    lerp(madd(t, x[0], f[0]), madd(t, x[1], f[2]), v[0][0], v[0][1]);
    lerp(madd(-t, x[0], f[1]), madd(-t, x[1], f[3]), v[1][0], v[1][1]);
  }
};

// Three times the sum over Gauss points of grad c . grad c (raw differences), a
// quadratic form with constant entries: the squared differences of the pairs of
// corners that differ in two or three axes (2D: in one, and twice those in two).
template <int D, class T>
__device__ __forceinline__ T grad_squares(const T* c) {
  T s = T(0);
#pragma unroll
  for (int a = 0; a < (1 << D); ++a)
#pragma unroll
    for (int b = a + 1; b < (1 << D); ++b) {
      const int n = ((a ^ b) & 1) + (((a ^ b) >> 1) & 1) + ((a ^ b) >> 2);
      if (D == 3 && n == 1) continue;
      const T d = c[b] - c[a];
      s = D == 2 && n == 2 ? madd(twice(d), d, s) : madd(d, d, s);
    }
  return s;
}
// Half the derivative of grad_squares: for each corner the differences to its
// partners (3/2 of the rows int grad c . grad phi in the same units).
template <int D, class T>
__device__ __forceinline__ void grad_rows(const T* c, T (&r)[1 << D]) {
  if constexpr (D == 3) {
    // to the opposite corner, and to those opposite in a face across x, y and z
    T body[4], fx[4], fy[4], fz[8];
#pragma unroll
    for (int a = 0; a < 4; ++a) {
      const int k = (a & 1) | (a & 2) << 1;  // 0, 1, 4, 5
      body[a] = c[a] - c[a ^ 7];
      fx[a] = c[a] - c[a ^ 6];
      fy[a] = c[a] - c[a ^ 5];
      fz[k] = c[k] - c[k ^ 3];
      fz[k ^ 3] = -fz[k];
    }
#pragma unroll
    for (int a = 0; a < 4; ++a) {
      const int o = a ^ 7;
      r[a] = (body[a] + fx[a]) + (fy[a] + fz[a]);
      r[o] = (fz[o] - body[a]) - (fx[o ^ 6] + fy[o ^ 5]);
    }
  } else {
    const T x0 = c[1] - c[0], x1 = c[3] - c[2], y0 = c[2] - c[0], y1 = c[3] - c[1];
    const T e = twice(c[3] - c[0]), f = twice(c[1] - c[2]);
    r[0] = -(e + (x0 + y0));
    r[1] = f + (x0 - y1);
    r[2] = (y0 - x1) - f;
    r[3] = e + (x1 + y1);
  }
}

// Energy of one element: sum_q w [g psi + Gc/2 (c^2/ls + ls |grad c|^2) + p g tr].
// With raw differences and 1/h folded into the constants,
//   psi + p tr = (lam/2 tr + p) tr + mu (sum of G_ii^2 + sum of (G_ik + G_ki)^2 / 2).
// tr and the symmetric sums are formed before they are squared: a quadratic in
// the single derivatives (lam/2 + mu) G_ii^2 + lam G_ii G_kk + ... cancels, its
// error grown by lam / mu where tr is small against them (1e-12 at nu =
// 0.499999) and by |rotation|^2 / |strain|^2.  A square G_ii^2 is shared by two
// Gauss points.  ROLL keeps the two z layers of Gauss points a loop (see the
// double-float kernels).
template <int D, class T, bool ROLL = false>
__device__ __forceinline__ T elem_energy(const T (*xe)[1 << D], const Mat<T>& m) {
  const T omk = T(1) - m.k, ih2 = m.inv_h * m.inv_h;
  const T hl = T(0.5) * m.lam * ih2, cm = m.mu * ih2, hcm = T(0.5) * cm;
  const T cp = m.p * m.inv_h;
  T acc = T(0), c2 = T(0);
  auto weighted = [&](T W, T cq, T sum) {
    const T o = T(1) - cq;
    c2 = madd(cq, cq, c2);
    return madd(madd(omk * o, o, m.k), W, sum);
  };
  if constexpr (D == 3) {
    Corners3<T, true> u[3], c;
#pragma unroll
    for (int i = 0; i < 3; ++i) u[i].set(xe[i]);
    c.set(xe[3]);
    T uz[3][2][2], C[2][2];
#pragma unroll
    for (int i = 0; i < 3; ++i) u[i].dz(uz[i]);
#pragma unroll
    for (int k = 0; k < 4; ++k) C[k & 1][k >> 1] = uz[2][k & 1][k >> 1] * uz[2][k & 1][k >> 1];
#pragma unroll (ROLL ? 1 : 2)
    for (int qz = 0; qz < 2; ++qz) {
      T ux[3][2], uy[3][2], v[2][2], A[2], B[2], sum = T(0);
#pragma unroll
      for (int i = 0; i < 3; ++i) u[i].dxy(qz, ux[i], uy[i]);
      c.values(qz, v);
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        A[k] = ux[0][k] * ux[0][k];
        B[k] = uy[1][k] * uy[1][k];
      }
#pragma unroll
      for (int qx = 0; qx < 2; ++qx)
#pragma unroll
        for (int qy = 0; qy < 2; ++qy) {
          const T tr = (ux[0][qy] + uy[1][qx]) + uz[2][qx][qy];
          const T s01 = ux[1][qy] + uy[0][qx], s02 = ux[2][qy] + uz[0][qx][qy], s12 = uy[2][qx] + uz[1][qx][qy];
          const T off = madd(s01, s01, madd(s02, s02, s12 * s12));
          const T W = madd(madd(hl, tr, cp), tr, madd(hcm, off, cm * ((A[qy] + B[qx]) + C[qx][qy])));
          sum = weighted(W, v[qx][qy], sum);
        }
      acc = acc + sum;
    }
  } else {
    Corners2<T> u[2], c;
    u[0].set(xe[0]);
    u[1].set(xe[1]);
    c.set(xe[2]);
    T ux[2][2], uy[2][2], v[2][2], A[2], B[2];
    u[0].dxy(ux[0], uy[0]);
    u[1].dxy(ux[1], uy[1]);
    c.values(v);
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      A[k] = ux[0][k] * ux[0][k];
      B[k] = uy[1][k] * uy[1][k];
    }
#pragma unroll
    for (int qx = 0; qx < 2; ++qx)
#pragma unroll
      for (int qy = 0; qy < 2; ++qy) {
        const T tr = ux[0][qy] + uy[1][qx], s01 = ux[1][qy] + uy[0][qx];
        const T W = madd(madd(hl, tr, cp), tr, madd(hcm * s01, s01, cm * (A[qy] + B[qx])));
        acc = weighted(W, v[qx][qy], acc);
      }
  }
  const T gr = (m.Gc * m.ls) * ih2 * T(1.0 / 3.0);
  return m.w * madd(T(0.5) * m.gcl, c2, madd(gr, grad_squares<D, T>(xe[D]), acc));
}

// What the gradient and the Hessian coefficients share at one Gauss point,
// from the raw differences G[i][k] of the displacement: t_i = (sigma + p I)_ii
// and t_ik = sigma_ik (physical), and W = (2 h) (psi + p tr).
template <int D, class T>
struct Point {
  T t[D], ts[D == 3 ? 3 : 1], W;
  __device__ __forceinline__ void set(const T (&G)[D][D], T lh, T mh, T mh2, T p) {
    T tr = G[0][0] + G[1][1];
    if constexpr (D == 3) tr = tr + G[D - 1][D - 1];
    const T dia = madd(lh, tr, p);
    W = p * tr;
#pragma unroll
    for (int i = 0; i < D; ++i) {
      t[i] = madd(mh2, G[i][i], dia);
      W = madd(t[i], G[i][i], W);
    }
#pragma unroll
    for (int i = 0; i < D; ++i)
#pragma unroll
      for (int k = i + 1; k < D; ++k) {
        const int j = sym_index<D>(i, k) - D;
        const T s = G[i][k] + G[k][i];
        ts[j] = mh * s;
        W = madd(ts[j], s, W);
      }
  }
};

// Strain invariants of a displacement gradient G (physical units):
// tr = div u, ee = eps : eps, and the symmetric off-diagonal sums
// G_ik + G_ki (i < k) in sym order 01, (02, 12).
template <int D, class T>
struct StrainSym {
  T tr, ee, off[D == 3 ? 3 : 1];
  __device__ __forceinline__ void set(const T G[D][D]) {
    tr = T(0);
    ee = T(0);
#pragma unroll
    for (int i = 0; i < D; ++i) {
      tr += G[i][i];
      ee += G[i][i] * G[i][i];
    }
#pragma unroll
    for (int i = 0; i < D; ++i)
#pragma unroll
      for (int k = i + 1; k < D; ++k) {
        const T sik = G[i][k] + G[k][i];
        off[sym_index<D>(i, k) - D] = sik;
        ee += T(0.5) * sik * sik;
      }
  }
};

// Quartic coefficients of E_e(x + t s) - E_e(x).  Gradients stay raw nodal
// differences; 1/h and 1/h^2 are folded into the constants.
template <int D, class T>
__device__ __forceinline__ void elem_energy_diff(const T (*xe)[1 << D], const T (*se)[1 << D],
                                                 const Mat<T>& m, T a[4]) {
  constexpr int NQ = 1 << D;
  T gu[D][D][NQ], cv[NQ], gc[D][NQ], dummy[NQ];
  T gs[D][D][NQ], sc[NQ], gsc[D][NQ];
#pragma unroll
  for (int i = 0; i < D; ++i) {
    interp<D, T>(xe[i], dummy, gu[i]);
    interp<D, T>(se[i], dummy, gs[i]);
  }
  interp<D, T>(xe[D], cv, gc);
  interp<D, T>(se[D], sc, gsc);
  T a1 = 0, a2 = 0, a3 = 0, a4 = 0;
  const T omk = T(1) - m.k;
  const T ih2 = m.inv_h * m.inv_h;
  const T hl = T(0.5) * m.lam * ih2, lam2 = m.lam * ih2, mu2 = m.mu * ih2, ph = m.p * m.inv_h;
  const T gls = m.Gc * m.ls * ih2, hgls = T(0.5) * gls, gcl = m.gcl, hgcl = T(0.5) * gcl;
#pragma unroll
  for (int q = 0; q < NQ; ++q) {
    T G[D][D], Gs[D][D];
#pragma unroll
    for (int i = 0; i < D; ++i)
#pragma unroll
      for (int k = 0; k < D; ++k) {
        G[i][k] = gu[i][k][q];
        Gs[i][k] = gs[i][k][q];
      }
    StrainSym<D, T> e0, e1;
    e0.set(G);
    e1.set(Gs);
    T e01 = T(0);  // eps(u) : eps(s), raw
#pragma unroll
    for (int i = 0; i < D; ++i) e01 += G[i][i] * Gs[i][i];
#pragma unroll
    for (int j = 0; j < (D == 3 ? 3 : 1); ++j) e01 += T(0.5) * e0.off[j] * e1.off[j];
    const T psi0 = hl * e0.tr * e0.tr + mu2 * e0.ee;
    const T psi2 = hl * e1.tr * e1.tr + mu2 * e1.ee;
    const T psi1 = lam2 * e0.tr * e1.tr + T(2) * mu2 * e01;
    const T omc = T(1) - cv[q], s = sc[q];
    const T g0 = omk * omc * omc + m.k;
    const T g1 = T(-2) * omk * omc * s;
    const T g2 = omk * s * s;
    T cg = 0, gg = 0;
#pragma unroll
    for (int k = 0; k < D; ++k) {
      const T u = gc[k][q], v = gsc[k][q];
      cg += u * v;
      gg += v * v;
    }
    const T t0 = ph * e0.tr, t1 = ph * e1.tr;
    a1 += g0 * psi1 + g1 * psi0 + (g0 * t1 + g1 * t0) + gcl * cv[q] * s + gls * cg;
    a2 += g0 * psi2 + g1 * psi1 + g2 * psi0 + (g1 * t1 + g2 * t0) + hgcl * s * s + hgls * gg;
    a3 += g1 * psi2 + g2 * psi1 + g2 * t1;
    a4 += g2 * psi2;
  }
  a[0] = m.w * a1; a[1] = m.w * a2; a[2] = m.w * a3; a[3] = m.w * a4;
}

// Gradient: u-rows  int g (sigma + p I) : grad phi,
//           c-row   int [g'(psi + p tr) + Gc c/ls] phi + Gc ls grad c . grad phi.
// The test functions' sums go axis by axis: an x-derivative row is summed
// over qx, weighted by N_ay, then by N_az, and enters the corners ax = 0, 1
// with opposite signs; the others likewise.

// N_0 and N_1 weighted sums of the two Gauss values along an axis
template <class T>
__device__ __forceinline__ void n_sums(T v0, T v1, T& n0, T& n1) {
  const T x0 = T(PF_XI0), x1 = T(PF_XI1);
  n0 = madd(x1, v0, x0 * v1);
  n1 = madd(x0, v0, x1 * v1);
}

// Sums of one field's derivative rows over a z layer of Gauss points.
template <class T>
struct Rows3 {
  T tx[2][2], ty[2][2], zs[2][2];  // [ay][az], [ax][az], [qx][qy]
  __device__ __forceinline__ void zero() {
#pragma unroll
    for (int i = 0; i < 4; ++i) tx[i & 1][i >> 1] = ty[i & 1][i >> 1] = zs[i & 1][i >> 1] = T(0);
  }
  // sx by qy (summed over qx), sy by qx (summed over qy), weights of az
  __device__ __forceinline__ void add_xy(T sx0, T sx1, T sy0, T sy1, T w0, T w1) {
    T a, b;
    n_sums(sx0, sx1, a, b);
    tx[0][0] = madd(w0, a, tx[0][0]);
    tx[0][1] = madd(w1, a, tx[0][1]);
    tx[1][0] = madd(w0, b, tx[1][0]);
    tx[1][1] = madd(w1, b, tx[1][1]);
    n_sums(sy0, sy1, a, b);
    ty[0][0] = madd(w0, a, ty[0][0]);
    ty[0][1] = madd(w1, a, ty[0][1]);
    ty[1][0] = madd(w0, b, ty[1][0]);
    ty[1][1] = madd(w1, b, ty[1][1]);
  }
  __device__ __forceinline__ void corners(T* r) {
    T tz[2][2];
    {
      T n[2][2];
      n_sums(zs[0][0], zs[1][0], n[0][0], n[1][0]);
      n_sums(zs[0][1], zs[1][1], n[0][1], n[1][1]);
      n_sums(n[0][0], n[0][1], tz[0][0], tz[0][1]);
      n_sums(n[1][0], n[1][1], tz[1][0], tz[1][1]);
    }
#pragma unroll
    for (int a = 0; a < 8; ++a) {
      const int ax = a & 1, ay = (a >> 1) & 1, az = a >> 2;
      T v = ax ? tx[ay][az] : -tx[ay][az];
      v = ay ? v + ty[ax][az] : v - ty[ax][az];
      r[a] = az ? v + tz[ax][ay] : v - tz[ax][ay];
    }
  }
};

template <int D, class T, bool ROLL = false>
__device__ __forceinline__ void elem_gradient(const T (*xe)[1 << D], const Mat<T>& m,
                                              T (*out)[1 << D]) {
  const T x0 = T(PF_XI0), x1 = T(PF_XI1);
  const T wh = m.w * m.inv_h, wo = wh * (T(1) - m.k), wk = wh * m.k, wc = m.w * m.gcl;
  const T lh = m.lam * m.inv_h, mh = m.mu * m.inv_h, mh2 = twice(mh);
  const T kc = wh * m.Gc * m.ls * m.inv_h * T(2.0 / 3.0);  // of grad_rows
  if constexpr (D == 3) {
    Corners3<T, !ROLL> u[3], c;
#pragma unroll
    for (int i = 0; i < 3; ++i) u[i].set(xe[i]);
    c.set(xe[3]);
    T uz[3][2][2];
#pragma unroll
    for (int i = 0; i < 3; ++i) u[i].dz(uz[i]);
    Rows3<T> r[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) r[i].zero();
    T s[8];  // row of c
    grad_rows<3, T>(xe[3], s);
#pragma unroll
    for (int i = 0; i < 8; ++i) s[i] = kc * s[i];
#pragma unroll (ROLL ? 1 : 2)
    for (int qz = 0; qz < 2; ++qz) {
      const T w0 = qz ? x0 : x1, w1 = qz ? x1 : x0;
      T ux[3][2], uy[3][2], v[2][2], s0[2][2];
      T sx[3][2], sy[3][2];  // by qy, by qx
#pragma unroll
      for (int i = 0; i < 3; ++i) u[i].dxy(qz, ux[i], uy[i]);
      c.values(qz, v);
#pragma unroll
      for (int qx = 0; qx < 2; ++qx)
#pragma unroll
        for (int qy = 0; qy < 2; ++qy) {
          T G[3][3];
#pragma unroll
          for (int i = 0; i < 3; ++i) {
            G[i][0] = ux[i][qy];
            G[i][1] = uy[i][qx];
            G[i][2] = uz[i][qx][qy];
          }
          Point<3, T> P;
          P.set(G, lh, mh, mh2, m.p);
          const T o = T(1) - v[qx][qy], q1 = wo * o, g = madd(q1, o, wk);
          s0[qx][qy] = madd(-q1, P.W, wc * v[qx][qy]);
          const T S01 = g * P.ts[0], S02 = g * P.ts[1], S12 = g * P.ts[2];
          const T S[3][3] = {{g * P.t[0], S01, S02}, {S01, g * P.t[1], S12}, {S02, S12, g * P.t[2]}};
#pragma unroll
          for (int i = 0; i < 3; ++i) {
            sx[i][qy] = qx ? sx[i][qy] + S[i][0] : S[i][0];
            sy[i][qx] = qy ? sy[i][qx] + S[i][1] : S[i][1];
            r[i].zs[qx][qy] = r[i].zs[qx][qy] + S[i][2];
          }
        }
#pragma unroll
      for (int i = 0; i < 3; ++i) r[i].add_xy(sx[i][0], sx[i][1], sy[i][0], sy[i][1], w0, w1);
      T n[2][2], nn[2][2];
      n_sums(s0[0][0], s0[1][0], n[0][0], n[1][0]);
      n_sums(s0[0][1], s0[1][1], n[0][1], n[1][1]);
      n_sums(n[0][0], n[0][1], nn[0][0], nn[0][1]);
      n_sums(n[1][0], n[1][1], nn[1][0], nn[1][1]);
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        s[i] = madd(w0, nn[i & 1][i >> 1], s[i]);
        s[i + 4] = madd(w1, nn[i & 1][i >> 1], s[i + 4]);
      }
    }
#pragma unroll
    for (int i = 0; i < 3; ++i) r[i].corners(out[i]);
#pragma unroll
    for (int a = 0; a < 8; ++a) out[3][a] = s[a];
  } else {
    Corners2<T> u[2], c;
    u[0].set(xe[0]);
    u[1].set(xe[1]);
    c.set(xe[2]);
    T ux[2][2], uy[2][2], v[2][2], s0[2][2], sx[2][2], sy[2][2];
    u[0].dxy(ux[0], uy[0]);
    u[1].dxy(ux[1], uy[1]);
    c.values(v);
#pragma unroll
    for (int qx = 0; qx < 2; ++qx)
#pragma unroll
      for (int qy = 0; qy < 2; ++qy) {
        const T G[2][2] = {{ux[0][qy], uy[0][qx]}, {ux[1][qy], uy[1][qx]}};
        Point<2, T> P;
        P.set(G, lh, mh, mh2, m.p);
        const T o = T(1) - v[qx][qy], q1 = wo * o, g = madd(q1, o, wk);
        s0[qx][qy] = madd(-q1, P.W, wc * v[qx][qy]);
        const T S01 = g * P.ts[0];
        const T S[2][2] = {{g * P.t[0], S01}, {S01, g * P.t[1]}};
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          sx[i][qy] = qx ? sx[i][qy] + S[i][0] : S[i][0];
          sy[i][qx] = qy ? sy[i][qx] + S[i][1] : S[i][1];
        }
      }
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      T a, b, e, f;
      n_sums(sx[i][0], sx[i][1], a, b);  // by ay
      n_sums(sy[i][0], sy[i][1], e, f);  // by ax
      out[i][0] = -a - e;
      out[i][1] = a - f;
      out[i][2] = e - b;
      out[i][3] = b + f;
    }
    T n[2][2], nn[2][2], d[4];
    n_sums(s0[0][0], s0[1][0], n[0][0], n[1][0]);
    n_sums(s0[0][1], s0[1][1], n[0][1], n[1][1]);
    n_sums(n[0][0], n[0][1], nn[0][0], nn[0][1]);
    n_sums(n[1][0], n[1][1], nn[1][0], nn[1][1]);
    grad_rows<2, T>(xe[2], d);
#pragma unroll
    for (int k = 0; k < 4; ++k) out[2][k] = madd(kc, d[k], nn[k & 1][k >> 1]);
  }
}

// Gradient difference grad E_e(x + s) - grad E_e(x), written so that every
// term is of order one or higher in s (no difference of two gradients is
// formed; for c' = c + s_c, u' = u + s_u):
//   u-rows  int [g(c') sigma(s_u) + (g(c') - g(c)) (sigma(u) + p I)] : grad phi
//   c-row   int [g'(c') (psi_1 + psi(s_u) + p tr s_u)
//                + (g'(c') - g'(c)) (psi(u) + p tr u) + Gc s_c/ls] phi
//               + Gc ls grad s_c . grad phi
// with psi_1 = lam tr(u) tr(s_u) + 2 mu eps(u) : eps(s_u),
// g(c') - g(c) = (1-k) s_c (s_c - 2 (1-c)) and g'(c') - g'(c) = 2 (1-k) s_c.
template <int D, class T>
__device__ __forceinline__ void elem_gradient_diff(const T (*xe)[1 << D], const T (*se)[1 << D],
                                                   const Mat<T>& m, T (*out)[1 << D]) {
  constexpr int NQ = 1 << D;
  T su[D][D][NQ], s0[NQ], sc[D][NQ];
  {
    T gu[D][D][NQ], cv[NQ], gcx[D][NQ], dummy[NQ];
    T gs[D][D][NQ], scv[NQ], gsc[D][NQ];
#pragma unroll
    for (int i = 0; i < D; ++i) {
      interp<D, T>(xe[i], dummy, gu[i]);
      interp<D, T>(se[i], dummy, gs[i]);
    }
    interp<D, T>(xe[D], cv, gcx);
    interp<D, T>(se[D], scv, gsc);
    const T omk = T(1) - m.k;
    const T kc = m.w * m.Gc * m.ls * m.inv_h * m.inv_h;
    const T gcl = m.gcl;
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
      T G[D][D], Gs[D][D];
#pragma unroll
      for (int i = 0; i < D; ++i)
#pragma unroll
        for (int k = 0; k < D; ++k) {
          G[i][k] = gu[i][k][q] * m.inv_h;
          Gs[i][k] = gs[i][k][q] * m.inv_h;
        }
      StrainSym<D, T> e0, e1;
      e0.set(G);
      e1.set(Gs);
      T e01 = T(0);
#pragma unroll
      for (int i = 0; i < D; ++i) e01 += G[i][i] * Gs[i][i];
#pragma unroll
      for (int j = 0; j < (D == 3 ? 3 : 1); ++j) e01 += T(0.5) * e0.off[j] * e1.off[j];
      const T psi0 = T(0.5) * m.lam * e0.tr * e0.tr + m.mu * e0.ee;
      const T psi2 = T(0.5) * m.lam * e1.tr * e1.tr + m.mu * e1.ee;
      const T psi1 = m.lam * e0.tr * e1.tr + T(2) * m.mu * e01;
      const T omc = T(1) - cv[q], sq = scv[q], omc1 = omc - sq;
      const T g1 = omk * omc1 * omc1 + m.k;         // g(c')
      const T dg = omk * sq * (sq - T(2) * omc);      // g(c') - g(c)
      const T dp1 = T(-2) * omk * omc1;               // g'(c')
      const T wg1 = m.w * m.inv_h * g1, wdg = m.w * m.inv_h * dg;
      const T d0 = m.lam * e0.tr + m.p, d1 = m.lam * e1.tr;
#pragma unroll
      for (int i = 0; i < D; ++i) {
        su[i][i][q] = wg1 * (d1 + T(2) * m.mu * Gs[i][i]) + wdg * (d0 + T(2) * m.mu * G[i][i]);
#pragma unroll
        for (int k = i + 1; k < D; ++k) {
          const int j = sym_index<D>(i, k) - D;
          const T v = m.mu * (wg1 * e1.off[j] + wdg * e0.off[j]);
          su[i][k][q] = v;
          su[k][i][q] = v;
        }
      }
      s0[q] = m.w * (dp1 * (psi1 + psi2 + m.p * e1.tr) + T(2) * omk * sq * (psi0 + m.p * e0.tr) +
                     gcl * sq);
#pragma unroll
      for (int k = 0; k < D; ++k) sc[k][q] = kc * gsc[k][q];
    }
  }
#pragma unroll
  for (int i = 0; i < D; ++i) test<D, T>(nullptr, su[i], out[i]);
  test<D, T>(s0, sc, out[D]);
}

// ---------------------------------------------------------------- Hessian
// The Hessian at x applied to v,
//   u-rows  int [g sigma(v_u) + g' v_c (sigma(u) + p I)] : grad phi
//   c-row   int [g' (sigma(u) + p I) : eps(v_u) + (g''(psi + p tr) + Gc/ls) v_c] phi
//               + Gc ls grad v_c . grad phi
// depends on x only through three Gauss-point coefficients (raw nodal
// differences for the gradients, 1/h and the weight folded in):
//   A = w g / h^2,   B = w g' (sigma(u) + p I) / h  (symmetric),
//   M = w (g''(psi + p tr) + Gc/ls).
// Under Hessian lagging they are computed once per lagged point and every
// Hessian-vector product then needs only the v-part below.
// cf[q][0] = A, cf[q][1] = M, cf[q][2 + s] = B_s
template <int D, class T>
__device__ __forceinline__ void hess_coef(const T (*xe)[1 << D], const Mat<T>& m,
                                          T (*cf)[NCoef<D>::value]) {
  const T omk = T(1) - m.k, wh = m.w * m.inv_h, wo = wh * omk, nwo2 = -twice(wo);
  const T a1 = wo * m.inv_h, a0 = wh * m.inv_h * m.k, wc = m.w * m.gcl;
  const T lh = m.lam * m.inv_h, mh = m.mu * m.inv_h, mh2 = twice(mh);
  auto point = [&](const T (&G)[D][D], T cq, T (&o)[NCoef<D>::value]) {
    Point<D, T> P;
    P.set(G, lh, mh, mh2, m.p);
    const T omc = T(1) - cq, dgw = nwo2 * omc;
    o[0] = madd(a1 * omc, omc, a0);
    o[1] = madd(wo, P.W, wc);
#pragma unroll
    for (int i = 0; i < D; ++i) {
      o[2 + i] = dgw * P.t[i];
#pragma unroll
      for (int k = i + 1; k < D; ++k)
        o[2 + sym_index<D>(i, k)] = dgw * P.ts[sym_index<D>(i, k) - D];
    }
  };
  if constexpr (D == 3) {
    Corners3<T, true> u[3], c;
#pragma unroll
    for (int i = 0; i < 3; ++i) u[i].set(xe[i]);
    c.set(xe[3]);
    T uz[3][2][2];
#pragma unroll
    for (int i = 0; i < 3; ++i) u[i].dz(uz[i]);
#pragma unroll
    for (int qz = 0; qz < 2; ++qz) {
      T ux[3][2], uy[3][2], v[2][2];
#pragma unroll
      for (int i = 0; i < 3; ++i) u[i].dxy(qz, ux[i], uy[i]);
      c.values(qz, v);
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int qx = q & 1, qy = q >> 1;
        T G[3][3];
#pragma unroll
        for (int i = 0; i < 3; ++i) {
          G[i][0] = ux[i][qy];
          G[i][1] = uy[i][qx];
          G[i][2] = uz[i][qx][qy];
        }
        point(G, v[qx][qy], cf[q + 4 * qz]);
      }
    }
  } else {
    Corners2<T> u[2], c;
    u[0].set(xe[0]);
    u[1].set(xe[1]);
    c.set(xe[2]);
    T ux[2][2], uy[2][2], v[2][2];
    u[0].dxy(ux[0], uy[0]);
    u[1].dxy(ux[1], uy[1]);
    c.values(v);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int qx = q & 1, qy = q >> 1;
      const T G[2][2] = {{ux[0][qy], uy[0][qx]}, {ux[1][qy], uy[1][qx]}};
      point(G, v[qx][qy], cf[q]);
    }
  }
}

// The v-part: out = H v from the coefficients of the element's Gauss points.
template <int D, class T>
__device__ __forceinline__ void hess_apply(const T (*ve)[1 << D], const T (*cf)[NCoef<D>::value],
                                           const Mat<T>& m, T (*out)[1 << D]) {
  constexpr int NQ = 1 << D;
  T su[D][D][NQ], s0[NQ], sc[D][NQ];
  {
    T gv[D][D][NQ], vc[NQ], gvc[D][NQ], dummy[NQ];
#pragma unroll
    for (int i = 0; i < D; ++i) interp<D, T>(ve[i], dummy, gv[i]);
    interp<D, T>(ve[D], vc, gvc);
    const T kc = m.w * m.Gc * m.ls * m.inv_h * m.inv_h;
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
        const T A = cf[q][0], M = cf[q][1];
      T trr = T(0);
#pragma unroll
      for (int i = 0; i < D; ++i) trr += gv[i][i][q];
      const T lt = m.lam * trr, am = A * m.mu;
      T c0 = M * vc[q];
#pragma unroll
      for (int i = 0; i < D; ++i) {
        const T Bii = cf[q][2 + i];
        su[i][i][q] = A * (lt + T(2) * m.mu * gv[i][i][q]) + vc[q] * Bii;
        c0 += Bii * gv[i][i][q];
#pragma unroll
        for (int k = i + 1; k < D; ++k) {
          const T Bik = cf[q][2 + sym_index<D>(i, k)];
          const T sik = gv[i][k][q] + gv[k][i][q];
          const T v = am * sik + vc[q] * Bik;
          su[i][k][q] = v;
          su[k][i][q] = v;
          c0 += Bik * sik;
        }
      }
      s0[q] = c0;
#pragma unroll
      for (int k = 0; k < D; ++k) sc[k][q] = kc * gvc[k][q];
    }
  }
#pragma unroll
  for (int i = 0; i < D; ++i) test<D, T>(nullptr, su[i], out[i]);
  test<D, T>(s0, sc, out[D]);
}

template <int D, class T>
__device__ __forceinline__ void elem_hessvec(const T (*xe)[1 << D], const T (*ve)[1 << D],
                                             const Mat<T>& m, T (*out)[1 << D]) {
  T cf[1 << D][NCoef<D>::value];
  hess_coef<D, T>(xe, m, cf);
  hess_apply<D, T>(ve, cf, m, out);
}

// Diagonal of the Hessian (Jacobi preconditioner):
//   u_i dof of corner a: sum_q w g [lam (d_i phi_a)^2 + mu (|grad phi_a|^2 + (d_i phi_a)^2)]
//   c dof:              sum_q w [(g''(psi + p tr) + Gc/ls) phi_a^2 + Gc ls |grad phi_a|^2]
template <int D, class T>
__device__ __forceinline__ void elem_hessdiag(const T (*xe)[1 << D], const Mat<T>& m,
                                              T (*out)[1 << D]) {
  constexpr int NQ = 1 << D;
  T gu[D][D][NQ], cv[NQ], gdummy[D][NQ], dummy[NQ];
#pragma unroll
  for (int i = 0; i < D; ++i) interp<D, T>(xe[i], dummy, gu[i]);
  interp<D, T>(xe[D], cv, gdummy);
  T gq[NQ], mq[NQ];
#pragma unroll
  for (int q = 0; q < NQ; ++q) {
    T G[D][D];
#pragma unroll
    for (int i = 0; i < D; ++i)
#pragma unroll
      for (int k = 0; k < D; ++k) G[i][k] = gu[i][k][q] * m.inv_h;
    Strain<D, T> e;
    e.set(G);
    const T psi = T(0.5) * m.lam * e.tr * e.tr + m.mu * e.ddot(e);
    const T omk = T(1) - m.k, omc = T(1) - cv[q];
    gq[q] = m.w * (omk * omc * omc + m.k);
    mq[q] = m.w * (T(2) * omk * (psi + m.p * e.tr) + m.gcl);
  }
  const T h2 = m.inv_h * m.inv_h;
#pragma unroll
  for (int a = 0; a < NQ; ++a) {
    T du[D], dc = T(0);
#pragma unroll
    for (int i = 0; i < D; ++i) du[i] = T(0);
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
      // 1D factors: N(q, a) = XI1 if q == a along the axis, else XI0
      T n1[D];
#pragma unroll
      for (int k = 0; k < D; ++k) n1[k] = (((q >> k) & 1) == ((a >> k) & 1)) ? T(PF_XI1) : T(PF_XI0);
      T phi = T(1);
#pragma unroll
      for (int k = 0; k < D; ++k) phi *= n1[k];
      T d2[D], g2 = T(0);
#pragma unroll
      for (int k = 0; k < D; ++k) {
        T t = T(1);
#pragma unroll
        for (int j = 0; j < D; ++j)
          if (j != k) t *= n1[j] * n1[j];
        d2[k] = t * h2;
        g2 += d2[k];
      }
#pragma unroll
      for (int i = 0; i < D; ++i) du[i] += gq[q] * (m.lam * d2[i] + m.mu * (g2 + d2[i]));
      dc += mq[q] * phi * phi + m.w * m.Gc * m.ls * g2;
    }
#pragma unroll
    for (int i = 0; i < D; ++i) out[i][a] = du[i];
    out[D][a] = dc;
  }
}

}  // namespace pf
