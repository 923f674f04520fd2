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
__device__ __forceinline__ float at(float2 v, int q) { return q ? v.y : v.x; }

// Raw-difference derivatives of one field: x by qy and y by qx (lanes qz), z by
// qy (lanes qx).
struct Grad {
  float2 x[2], y[2], z[2];
  // of a rough field (the direction: any nodal noise), differences along an
  // axis first and then the other two axes; smooth fields lose nothing
  __device__ __forceinline__ void rough(const float f[8]) {
    lerp2(lerp2(f[1] - f[0], f[5] - f[4]), lerp2(f[3] - f[2], f[7] - f[6]), x);
    lerp2(lerp2(f[2] - f[0], f[6] - f[4]), lerp2(f[3] - f[1], f[7] - f[5]), y);
    lerp2(lerp2(f[4] - f[0], f[5] - f[1]), lerp2(f[6] - f[2], f[7] - f[3]), z);
  }
  // of a smooth one, through its monomials
  __device__ __forceinline__ void smooth(const float f[8]) {
    const float2 x0 = bc(float(PF_XI0)), x1 = bc(float(PF_XI1));
    Mono3<float> m;
    m.set(f);
    const float2 a = pair(m.xz, m.x), a2 = pair(m.yz, m.y), b = pair(m.xyz, m.xy);
    x[0] = fma2(x0, b, a);
    x[1] = fma2(x1, b, a);
    y[0] = fma2(x0, b, a2);
    y[1] = fma2(x1, b, a2);
    const float2 c = pair(m.yz, m.z), d = pair(m.xyz, m.xz);  // by qy
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
// row by qy, lanes qx (summed over qz); with VALUE a value row [qx][qy], lanes
// qz.
template <bool VALUE>
__device__ __forceinline__ void corners(const float2 (&sx)[2], const float2 (&sy)[2], const float2 (&sz)[2],
                                        const float2 (&s0)[2][2], float (&r)[8]) {
  const float x0 = float(PF_XI0), x1 = float(PF_XI1);
  float2 t0, t1, u0, u1, l[4];  // l: corners of a layer, lanes qz (0: negative)
  n_sums2(sx[0], sx[1], t0, t1);
  n_sums2(sy[0], sy[1], u0, u1);
  l[0] = add2(t0, u0);
  l[1] = sub2(t0, u1);
  l[2] = sub2(u0, t1);
  l[3] = add2(t1, u1);
  if constexpr (VALUE) {
    float2 n[2][2], v[2];
    n_sums2(s0[0][0], s0[1][0], n[0][0], n[1][0]);
    n_sums2(s0[0][1], s0[1][1], n[0][1], n[1][1]);
    n_sums2(n[0][0], n[0][1], v[0], v[1]);
    l[0] = sub2(l[0], v[0]);
    l[2] = add2(l[2], v[1]);
    n_sums2(n[1][0], n[1][1], v[0], v[1]);
    l[1] = add2(l[1], v[0]);
    l[3] = add2(l[3], v[1]);
  }
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

// The 3D FP32 Hessian product of one element, bound by the FP32 pipe and the
// issue slots: 1,050 operations (an FFMA2 counts as two), by
// - the state in monomials (Mono3), the direction and the adjoint axis by axis;
// - raw differences and stresses in units of mu / h, t_ik = (sigma + p I)_ik
//   h / mu, so that shear stresses are the sums G_ik + G_ki themselves;
// - the cross terms through t instead of the coefficient tensor B = g' t:
//   q = g' w, su = A sigma(v) + q t, s0 = M w + g' t : grad v;
// in pairs of Gauss points along z, whose lanes the z passes fill and take
// apart by themselves (only the z-derivatives, the same at both, are copied).
// With pairs along x, interpolation passes and the coefficient tensor it was
// 1,310, and the element pass at 129^3 took 100 us, now 88.  In
// monomials throughout, both ways, it would be 930, but the rounding of a
// rough direction then grows twofold.
__device__ __forceinline__ void elem_hessvec(const float (*xe)[8], const float (*ve)[8],
                                             const Mat<float>& m, float (*out)[8]) {
  Grad u[3], v[3], w;
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    u[i].smooth(xe[i]);
    v[i].rough(ve[i]);
  }
  w.rough(ve[3]);
  float2 ov[2][2], wv[2][2];  // 1 - c and w at [qx][qy]
  {
    float2 o[4], e0[2], e1[2];
#pragma unroll
    for (int k = 0; k < 4; ++k) o[k] = lerp2(1.f - xe[3][k], 1.f - xe[3][k + 4]);
    lerp2(o[0], o[1], e0);
    lerp2(o[2], o[3], e1);
    lerp2(e0[0], e1[0], ov[0]);
    lerp2(e0[1], e1[1], ov[1]);
    lerp2(lerp2(ve[3][0], ve[3][4]), lerp2(ve[3][1], ve[3][5]), e0);
#pragma unroll
    for (int qx = 0; qx < 2; ++qx) {
      wv[qx][0] = fma2(w.y[qx], bc(float(PF_XI0)), e0[qx]);
      wv[qx][1] = fma2(w.y[qx], bc(float(PF_XI1)), e0[qx]);
    }
  }
  const float omk = 1.f - m.k;
  const float kap = m.w * m.mu * m.inv_h * m.inv_h, ko = kap * omk, kk = kap * m.k;
  const float pm = m.p * m.hmu, wg = m.w * m.gcl;
  // a derivative of w stands for two Gauss points
  const float kc = 2.f * m.w * m.Gc * m.ls * m.inv_h * m.inv_h;
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
  for (int i = 0; i < 3; ++i) corners<false>(sx[i], sy[i], sz[i], s0, out[i]);
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    w.x[k] = mul2(bc(kc), w.x[k]);
    w.y[k] = mul2(bc(kc), w.y[k]);
    w.z[k] = mul2(bc(kc), w.z[k]);
  }
  corners<true>(w.x, w.y, w.z, s0, out[3]);
}

}  // namespace p2
}  // namespace pf
