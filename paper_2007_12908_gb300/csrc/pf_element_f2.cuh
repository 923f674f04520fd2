// Packed FP32 variant of the 3D Q1 Hessian-vector element operation on the
// paired FP32 FMA/ADD/MUL instructions of sm_100+ (__ffma2_rn etc.): the two
// Gauss points of a pair along z are the lanes of a float2.
#pragma once
#include <cuda_runtime.h>

#include "pf_element.cuh"

namespace pf {
namespace p2 {

__device__ __forceinline__ float2 bc(float a) { return make_float2(a, a); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
// a - b, exact: b * (-1) + a rounds once
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __ffma2_rn(b, bc(-1.f), a); }

__device__ __forceinline__ float2 pair(float b, float a) {  // a + xi b at the two points of an axis
  return make_float2(fmaf(float(PF_XI0), b, a), fmaf(float(PF_XI1), b, a));
}

// The two Gauss points between a and b, each from its nearer end: the rounding
// of b - a enters with weight 0.21 at both.
__device__ __forceinline__ float2 lerp2(float a, float b) {
  const float x0 = float(PF_XI0), t = b - a;
  return make_float2(fmaf(x0, t, a), fmaf(-x0, t, b));
}
__device__ __forceinline__ void lerp2(float2 a, float2 b, float2 (&o)[2]) {
  const float2 t = sub2(b, a);
  o[0] = fma2(bc(float(PF_XI0)), t, a);
  o[1] = fma2(bc(-float(PF_XI0)), t, b);
}
// Values at [qx][qy] of those by corner of a layer.
__device__ __forceinline__ void lerp4(const float2 (&c)[4], float2 (&o)[2][2]) {
  float2 e0[2], e1[2];
  lerp2(c[0], c[1], e0);
  lerp2(c[2], c[3], e1);
  lerp2(e0[0], e1[0], o[0]);
  lerp2(e0[1], e1[1], o[1]);
}
__device__ __forceinline__ float at(float2 v, int q) { return q ? v.y : v.x; }

// Raw-difference derivatives of one field: x by qy and y by qx (lanes qz), z by
// qy (lanes qx).
struct Grad {
  float2 x[2], y[2], z[2];
  // the direction (any nodal noise): differences along an axis first, then the
  // other two axes
  __device__ __forceinline__ void direction(const float f[8]) {
    lerp2(lerp2(f[1] - f[0], f[5] - f[4]), lerp2(f[3] - f[2], f[7] - f[6]), x);
    lerp2(lerp2(f[2] - f[0], f[6] - f[4]), lerp2(f[3] - f[1], f[7] - f[5]), y);
    lerp2(lerp2(f[4] - f[0], f[5] - f[1]), lerp2(f[6] - f[2], f[7] - f[3]), z);
  }
  // the state: near ends along z, monomials in the other two axes
  __device__ __forceinline__ void state(const float f[8]) {
    const float2 x0 = bc(float(PF_XI0)), x1 = bc(float(PF_XI1));
    const float x00 = f[1] - f[0], x10 = f[3] - f[2], x01 = f[5] - f[4], x11 = f[7] - f[6];
    const float2 ax = lerp2(x00, x01), ay = lerp2(f[2] - f[0], f[6] - f[4]), b = lerp2(x10 - x00, x11 - x01);
    x[0] = fma2(x0, b, ax);
    x[1] = fma2(x1, b, ax);
    y[0] = fma2(x0, b, ay);
    y[1] = fma2(x1, b, ay);
    const float2 c = lerp2(f[4] - f[0], f[6] - f[2]), d = lerp2(x01 - x00, x11 - x10);  // by qy
    z[0] = pair(d.x, c.x);
    z[1] = pair(d.y, c.y);
  }
};

// N_0 and N_1 weighted sums along an axis
__device__ __forceinline__ void n_sums2(float2 a, float2 b, float2& n0, float2& n1) {
  const float2 x0 = bc(float(PF_XI0)), x1 = bc(float(PF_XI1));
  n0 = fma2(x1, a, mul2(x0, b));
  n1 = fma2(x0, a, mul2(x1, b));
}

// Test-function sums of one field: an x-derivative row by qy (summed over qx)
// and a y-derivative row by qx (summed over qy), lanes qz, and a z-derivative
// row by qy, lanes qx (summed over qz).
__device__ __forceinline__ void corners(const float2 (&sx)[2], const float2 (&sy)[2], const float2 (&sz)[2],
                                        float (&r)[8]) {
  const float x0 = float(PF_XI0), x1 = float(PF_XI1);
  float2 t0, t1, u0, u1, l[4];  // l: corners of a layer, lanes qz (0: negative)
  n_sums2(sx[0], sx[1], t0, t1);
  n_sums2(sy[0], sy[1], u0, u1);
  l[0] = add2(t0, u0);
  l[1] = sub2(t0, u1);
  l[2] = sub2(u0, t1);
  l[3] = add2(t1, u1);
  float2 n[2];
  n_sums2(sz[0], sz[1], n[0], n[1]);
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    float a, b;
    n_sums(n[k >> 1].x, n[k >> 1].y, a, b);
    const float t = k & 1 ? b : a, s = k ? 1.f : -1.f;
    r[k] = fmaf(s * x1, l[k].x, fmaf(s * x0, l[k].y, -t));
    r[k + 4] = fmaf(s * x0, l[k].x, fmaf(s * x1, l[k].y, t));
  }
}

// r = scale r + the sums of a value row [qx][qy], lanes qz.
__device__ __forceinline__ void add_values(const float2 (&s)[2][2], float scale, float (&r)[8]) {
  const float x0 = float(PF_XI0), x1 = float(PF_XI1);
  float2 n[2][2], v[4];
  n_sums2(s[0][0], s[1][0], n[0][0], n[1][0]);
  n_sums2(s[0][1], s[1][1], n[0][1], n[1][1]);
  n_sums2(n[0][0], n[0][1], v[0], v[2]);
  n_sums2(n[1][0], n[1][1], v[1], v[3]);
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    r[k] = fmaf(x1, v[k].x, fmaf(x0, v[k].y, scale * r[k]));
    r[k + 4] = fmaf(x0, v[k].x, fmaf(x1, v[k].y, scale * r[k + 4]));
  }
}

// The 3D FP32 Hessian product of one element, bound by the FP32 pipe and the
// issue slots: about 1,020 operations (an FFMA2 counts as two), by
// - raw differences and stresses in units of mu / h, t_ik = (sigma + p I)_ik
//   h / mu, so that shear stresses are the sums G_ik + G_ki themselves;
// - the cross terms through t instead of the coefficient tensor B = g' t:
//   q = g' w, su = A sigma(v) + q t, s0 = M w + g' t : grad v;
// - grad w . grad phi from corner differences (grad_rows);
// in pairs of Gauss points along z, whose lanes the z passes fill and take
// apart by themselves (only the z-derivatives, the same at both, are copied).
// With pairs along x, interpolation passes and the coefficient tensor it was
// 1,310, and the element pass at 129^3 took 100 us, now 91.  In
// monomials throughout, both ways, it would be 930, but the rounding of a
// rough direction then grows twofold; with the state alone as monomials in all
// three axes the c rows of a rough state had 1.15 times the error (1.80e-7
// against 1.57e-7 where the displacement terms decide), and the product took
// 103.1 us instead of 105.9.
__device__ __forceinline__ void elem_hessvec(const float (*xe)[8], const float (*ve)[8],
                                             const Mat<float>& m, float (*out)[8]) {
  Grad u[3], v[3];
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    u[i].state(xe[i]);
    v[i].direction(ve[i]);
  }
  float2 ov[2][2], wv[2][2];  // 1 - c and w at [qx][qy]
  {
    float2 o[4], w[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      o[k] = lerp2(1.f - xe[3][k], 1.f - xe[3][k + 4]);
      w[k] = lerp2(ve[3][k], ve[3][k + 4]);
    }
    lerp4(o, ov);
    lerp4(w, wv);
  }
  const float omk = 1.f - m.k;
  const float kap = m.w * m.mu * m.inv_h * m.inv_h, ko = kap * omk, kk = kap * m.k;
  const float pm = m.p * m.hmu, wg = m.w * m.gcl;
  const float2 lmu = bc(m.lmu), two = bc(2.f);
  float2 sx[3][2], sy[3][2], sz[3][2], s0[2][2];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int qx = q & 1, qy = q >> 1;
    float2 G[3][3], V[3][3];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      G[i][0] = u[i].x[qy];
      G[i][1] = u[i].y[qx];
      G[i][2] = bc(at(u[i].z[qy], qx));
      V[i][0] = v[i].x[qy];
      V[i][1] = v[i].y[qx];
      V[i][2] = bc(at(v[i].z[qy], qx));
    }
    const float2 tr = add2(add2(G[0][0], G[1][1]), G[2][2]);
    const float2 trv = add2(add2(V[0][0], V[1][1]), V[2][2]);
    const float2 dia = fma2(lmu, tr, bc(pm)), lt = mul2(lmu, trv);
    const float2 q1 = mul2(bc(ko), ov[qx][qy]);
    const float2 A = fma2(q1, ov[qx][qy], bc(kk));
    const float2 dg = mul2(bc(-2.f), q1), qw = mul2(dg, wv[qx][qy]);
    float2 S[3][3];
    float2 W = mul2(bc(pm), tr), dot;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      const float2 t = fma2(two, G[i][i], dia);
      W = fma2(t, G[i][i], W);
      dot = i ? fma2(t, V[i][i], dot) : mul2(t, V[i][i]);
      S[i][i] = fma2(A, fma2(two, V[i][i], lt), mul2(qw, t));
    }
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int k = i + 1; k < 3; ++k) {
        const float2 t = add2(G[i][k], G[k][i]), tv = add2(V[i][k], V[k][i]);
        W = fma2(t, t, W);
        dot = fma2(t, tv, dot);
        S[i][k] = S[k][i] = fma2(A, tv, mul2(qw, t));
      }
    // Gauss weight times 2 (1 - k) (psi + p tr) + Gc / ls
    const float2 M = fma2(bc(ko), W, bc(wg));
    s0[qx][qy] = fma2(dg, dot, mul2(M, wv[qx][qy]));
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      sx[i][qy] = qx ? add2(sx[i][qy], S[i][0]) : S[i][0];
      sy[i][qx] = qy ? add2(sy[i][qx], S[i][1]) : S[i][1];
      const float z = S[i][2].x + S[i][2].y;
      if (qx) sz[i][qy].y = z;
      else sz[i][qy].x = z;
    }
  }
#pragma unroll
  for (int i = 0; i < 3; ++i) corners(sx[i], sy[i], sz[i], out[i]);
  grad_rows<3, float>(ve[3], out[3]);
  add_values(s0, m.w * m.Gc * m.ls * m.inv_h * m.inv_h * float(2.0 / 3.0), out[3]);
}

}  // namespace p2
}  // namespace pf
