// Assembly of a lagged Hessian into its 3^d-point block stencil (Sec. 4.2.1:
// Hessians are assembled once per lag and applied many times): the FP64
// Hessian of a level from its Gauss-point coefficients, and the FP32 Galerkin
// operator of a coarse level from its stored coefficient moments
// (pf_galerkin.cu).
//
// FP64 runs at 2 lanes per SM and clock here, so the assembly is bound by
// its FP64 instruction count.  One thread per (node, offset) block that
// summed shape-function products over the Gauss points of every corner pair
// spent about 40,000 FP64 instructions per element (12.3 ms on 65 x 49 x 57
// nodes, pipe 90 % busy); everything that sum needs of an element is 252
// moments (43 in 2D) of its Gauss-point coefficients A, M and B, each a
// product of 1D factors:
//   NN_c  N_a N_b along an axis, c = a + b in {0, 1, 2}
//   N_b   where the other function is differentiated (a sign, +-1)
//   1     where both are
// so the moments are formed axis by axis (about 1,000 instructions per
// element) and a corner pair's 4 x 4 block is then 41 FMAs of moments with
// +-lam, +-mu, +-1.  Blocks of offsets o and -o are transposes: only the 14
// offsets up to the centre (5 in 2D) are formed and each is written twice.
//
// A CTA owns a tile of nodes (8 x 4 in 3D, 32 in 2D) and marches along the
// last axis, one element layer at a time: (1) the moments of the layer's
// 9 x 5 (33) elements go to shared memory, (2) each warp adds the pairs of
// its offsets.  A block with no offset along the march axis gets the pairs
// of two layers; its partial sum waits in shared memory.  Every sum has a
// fixed order and every entry is written once: no atomics, no clearing.
// 12.3 -> 1.42 ms on 65 x 49 x 57 nodes (FP64 pipe 82 % busy, 20.7 M warp
// instructions), 33 -> 15 us on 69 x 45.
#include <algorithm>
#include <cmath>

#include "pf_internal.h"

namespace pf {

namespace {

constexpr double X0 = PF_XI0, X1 = PF_XI1;

template <int D, class T>
struct Asm {
  static constexpr int F = D + 1;
  static constexpr int TX = D == 3 ? 8 : 32, TY = D == 3 ? 4 : 1;  // nodes of a tile layer (32)
  static constexpr int EX = TX + 1, EY = D == 3 ? TY + 1 : 1, E = EX * EY;
  static constexpr int WARPS = D == 3 ? 8 : 4, THREADS = 32 * WARPS;
  // CTAs per SM by registers (and, for doubles in 3D, shared memory)
  static constexpr int PER_SM = sizeof(T) == 4 ? (D == 3 ? 3 : 5) : (D == 3 ? 2 : 3);
  static constexpr int CARRY = D == 3 ? 5 : 2;    // of them, those along no march axis
  // first moment of each family
  static constexpr int DD = 0;                             // axis k: 3^(D-1) each
  static constexpr int NW = D == 3 ? 9 : 3;                // 3^(D-1)
  static constexpr int DN = DD + D * NW;                   // axis pair: 4 * 3^(D-2) each
  static constexpr int NDN = D == 3 ? 12 : 4, PAIRS = D == 3 ? 3 : 1;
  static constexpr int BB = DN + PAIRS * NDN;              // (i, k): 2 * 3^(D-1) each
  static constexpr int MM = BB + D * D * 2 * NW;           // 3^D
  static constexpr int COUNT = MM + 3 * NW;
  static constexpr int ROWS = COUNT + 1;                   // + the element's kc (0 outside)
  // phase-1 work in units of warps
  static constexpr int W_DD = (D * E + 31) / 32, W_DN = (PAIRS * E + 31) / 32;
  static constexpr int W_BB = (D * D * E + 31) / 32, W_MM = (E + 31) / 32;
  static constexpr int W_ALL = W_DD + W_DN + W_BB + W_MM;
  static constexpr size_t smem = sizeof(T) * (size_t(ROWS) * E + size_t(CARRY) * F * F * 32);
};

// NN_0, NN_1, NN_2 of the two Gauss values along an axis: x1^2 v0 + x0^2 v1,
// x0 x1 (v0 + v1) and x0^2 v0 + x1^2 v1, with x1^2 - x0^2 = x1 - x0
__device__ __forceinline__ void w3(double v0, double v1, double (&o)[3]) {
  const double s = v0 + v1, p = (X1 * X1) * s;
  o[0] = fma(X0 - X1, v1, p);
  o[1] = (X0 * X1) * s;
  o[2] = fma(X0 - X1, v0, p);
}
// N_0, N_1
__device__ __forceinline__ void n2(double v0, double v1, double (&o)[2]) {
  const double d = v1 - v0;
  o[0] = fma(X0, d, v0);
  o[1] = fma(X1, d, v0);
}

// The axes other than k, ascending.
__device__ __forceinline__ int other(int k, int j) { return j < k ? j : j + 1; }

// Moments of one family of one element: the 2^D Gauss values of coefficient
// `comp` with the axes taken in the order (k0, k1, k2), to out[m * E].
template <int D>
__device__ __forceinline__ void load_q(const double* __restrict__ coef, long long NE, long long e,
                                       bool in, int comp, int k0, int k1, int k2,
                                       double (&v)[1 << D]) {
  using A = Asm<D, double>;
#pragma unroll
  for (int q = 0; q < (1 << D); ++q) {
    int p = ((q & 1) << k0) | (((q >> 1) & 1) << k1);
    if (D == 3) p |= ((q >> 2) & 1) << k2;
    v[q] = in ? coef[((long long)p * NCoef<D>::value + comp) * NE + e] : 0.0;
  }
}

template <int D>
__device__ __forceinline__ void moments_dd(const double (&v)[1 << D], double* out) {
  constexpr int E = Asm<D, double>::E;
  if constexpr (D == 3) {
    double t[2][3];  // [v][p]
#pragma unroll
    for (int z = 0; z < 2; ++z) w3(v[4 * z] + v[4 * z + 1], v[4 * z + 2] + v[4 * z + 3], t[z]);
#pragma unroll
    for (int p = 0; p < 3; ++p) {
      double o[3];
      w3(t[0][p], t[1][p], o);
#pragma unroll
      for (int r = 0; r < 3; ++r) out[(p * 3 + r) * E] = o[r];
    }
  } else {
    double o[3];
    w3(v[0] + v[1], v[2] + v[3], o);
#pragma unroll
    for (int p = 0; p < 3; ++p) out[p * E] = o[p];
  }
}

template <int D>
__device__ __forceinline__ void moments_dn(const double (&v)[1 << D], double* out) {
  constexpr int E = Asm<D, double>::E, NZ = D == 3 ? 2 : 1;
  double m[NZ][2][2];  // [t][beta][alpha]
#pragma unroll
  for (int z = 0; z < NZ; ++z) {
    double a[2], b[2];
    n2(v[4 * z], v[4 * z + 1], a);
    n2(v[4 * z + 2], v[4 * z + 3], b);
#pragma unroll
    for (int be = 0; be < 2; ++be) n2(a[be], b[be], m[z][be]);
  }
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    if constexpr (D == 3) {
      double o[3];
      w3(m[0][k >> 1][k & 1], m[NZ - 1][k >> 1][k & 1], o);
#pragma unroll
      for (int r = 0; r < 3; ++r) out[(k * 3 + r) * E] = o[r];
    } else {
      out[k * E] = m[0][k >> 1][k & 1];
    }
  }
}

template <int D>
__device__ __forceinline__ void moments_b(const double (&v)[1 << D], double* out) {
  constexpr int E = Asm<D, double>::E, NW = Asm<D, double>::NW, NZ = D == 3 ? 2 : 1;
  double n[NZ][2][2];  // [v][u][beta]
#pragma unroll
  for (int z = 0; z < NZ; ++z)
#pragma unroll
    for (int u = 0; u < 2; ++u) n2(v[4 * z + 2 * u], v[4 * z + 2 * u + 1], n[z][u]);
#pragma unroll
  for (int be = 0; be < 2; ++be) {
    double t[NZ][3];
#pragma unroll
    for (int z = 0; z < NZ; ++z) w3(n[z][0][be], n[z][1][be], t[z]);
#pragma unroll
    for (int p = 0; p < 3; ++p) {
      if constexpr (D == 3) {
        double o[3];
        w3(t[0][p], t[NZ - 1][p], o);
#pragma unroll
        for (int r = 0; r < 3; ++r) out[(be * NW + p * 3 + r) * E] = o[r];
      } else {
        out[(be * NW + p) * E] = t[0][p];
      }
    }
  }
}

template <int D>
__device__ __forceinline__ void moments_m(const double (&v)[1 << D], double* out) {
  constexpr int E = Asm<D, double>::E, NZ = D == 3 ? 2 : 1;
  double x[NZ][2][3];
#pragma unroll
  for (int z = 0; z < NZ; ++z)
#pragma unroll
    for (int y = 0; y < 2; ++y) w3(v[4 * z + 2 * y], v[4 * z + 2 * y + 1], x[z][y]);
#pragma unroll
  for (int p = 0; p < 3; ++p) {
    double t[NZ][3];
#pragma unroll
    for (int z = 0; z < NZ; ++z) w3(x[z][0][p], x[z][1][p], t[z]);
#pragma unroll
    for (int r = 0; r < 3; ++r) {
      if constexpr (D == 3) {
        double o[3];
        w3(t[0][r], t[NZ - 1][r], o);
#pragma unroll
        for (int s = 0; s < 3; ++s) out[(p * 9 + r * 3 + s) * E] = o[s];
      } else {
        out[(p * 3 + r) * E] = t[0][r];
      }
    }
  }
}

// Adds corner pair (a, b) of the element whose moments start at mom: row
// fields at corner a, column fields at corner b.  The signs pick between a
// constant and its negative: a product with +-1 would be an FP64 instruction
// like any other (twice the pipe's work per pair).
template <class T>
struct PairConst {
  T lam, nlam, mu, nmu, l2m, nl2m;  // lam, mu, lam + 2 mu and their negatives
};
template <int D, class T>
__device__ __forceinline__ void add_pair(const T* __restrict__ mom, int a, int b,
                                         const PairConst<T>& C, T (&t)[(D + 1) * (D + 1)]) {
  using A = Asm<D, T>;
  constexpr int F = A::F, E = A::E;
  int ak[3], bk[3], c[3];
#pragma unroll
  for (int k = 0; k < D; ++k) {
    ak[k] = (a >> k) & 1;
    bk[k] = (b >> k) & 1;
    c[k] = ak[k] + bk[k];
  }
  // both differentiated along k: X_kk
#pragma unroll
  for (int k = 0; k < D; ++k) {
    const int u = other(k, 0), v = D == 3 ? other(k, 1) : 0;
    const int idx = D == 3 ? c[u] * 3 + c[v] : c[u];
    const T m = mom[(A::DD + k * A::NW + idx) * E];
    const bool same = ak[k] == bk[k];
    const T mu = same ? C.mu : C.nmu, lm = same ? C.l2m : C.nl2m;
#pragma unroll
    for (int i = 0; i < D; ++i) t[i * F + i] = fma(i == k ? lm : mu, m, t[i * F + i]);
  }
  // differentiated along k at a and l at b, and the other way round; the
  // sign is the product of the two corners' signs along those axes
#pragma unroll
  for (int k = 0; k < D; ++k)
#pragma unroll
    for (int l = k + 1; l < D; ++l) {
      const int pair = k + l - 1, r = D == 3 ? c[3 - k - l] : 0;
      const T* m = mom + (A::DN + pair * A::NDN) * E;
      const int nr = D == 3 ? 3 : 1;
      const T kl = m[((bk[k] * 2 + ak[l]) * nr + r) * E];  // X_kl
      const T lk = m[((ak[k] * 2 + bk[l]) * nr + r) * E];  // X_lk
      const bool p1 = ak[k] == bk[l], p2 = ak[l] == bk[k];
      const T lam1 = p1 ? C.lam : C.nlam, mu1 = p1 ? C.mu : C.nmu;
      const T lam2 = p2 ? C.lam : C.nlam, mu2 = p2 ? C.mu : C.nmu;
      t[k * F + l] = fma(lam1, kl, fma(mu2, lk, t[k * F + l]));
      t[l * F + k] = fma(lam2, lk, fma(mu1, kl, t[l * F + k]));
    }
  // displacement - phase field
#pragma unroll
  for (int i = 0; i < D; ++i)
#pragma unroll
    for (int k = 0; k < D; ++k) {
      const int u = other(k, 0), v = D == 3 ? other(k, 1) : 0;
      const int idx = D == 3 ? c[u] * 3 + c[v] : c[u];
      const T* m = mom + (A::BB + (i * D + k) * 2 * A::NW) * E;
      t[i * F + D] = fma(ak[k] ? T(1) : T(-1), m[(bk[k] * A::NW + idx) * E], t[i * F + D]);
      t[D * F + i] = fma(bk[k] ? T(1) : T(-1), m[(ak[k] * A::NW + idx) * E], t[D * F + i]);
    }
  // phase field; grad c . grad c has a constant coefficient, so its sum of
  // 1D products (2 where both are differentiated, else 2/3 for a = b along
  // the axis and 1/3 for a != b) depends on the number of axes with a != b
  const int im = D == 3 ? c[0] * 9 + c[1] * 3 + c[2] : c[0] * 3 + c[1];
  const int d = __popc(a ^ b);
  const T gg = D == 3 ? (d == 0 ? T(8.0 / 3.0) : (d == 1 ? T(0) : T(-2.0 / 3.0)))
                      : (d == 0 ? T(8.0 / 3.0) : (d == 1 ? T(-2.0 / 3.0) : T(-4.0 / 3.0)));
  t[D * F + D] = fma(gg, mom[A::COUNT * E], t[D * F + D] + mom[(A::MM + im) * E]);
}

// Offsets formed: the centre, then those with a positive last nonzero
// component; 2D ones have their march component in y.
template <int D>
__device__ __forceinline__ void half_offset(int j, int (&o)[3]) {
  if constexpr (D == 3) {
    // centre, x, y, xy, -x y, then (x, y, +1)
    const int x[14] = {0, 1, 0, 1, -1, 0, 1, -1, 0, 0, 1, -1, 1, -1};
    const int y[14] = {0, 0, 1, 1, 1, 0, 0, 0, 1, -1, 1, 1, -1, -1};
    o[0] = 0; o[1] = 0; o[2] = j >= 5 ? 1 : 0;
#pragma unroll
    for (int i = 0; i < 14; ++i)
      if (i == j) {
        o[0] = x[i];
        o[1] = y[i];
      }
  } else {
    o[0] = j == 1 || j == 3 ? 1 : (j == 4 ? -1 : 0);  // centre, x, y, xy, -x y
    o[1] = j >= 2 ? 1 : 0;
    o[2] = 0;
  }
}

// Offsets of a warp, [first, last): about as many pairs for each.
template <int D>
__device__ __forceinline__ int warp_offset(int warp, int n) {
  if constexpr (D == 3) {
    // 0 | 1 | 2 | 5 | 3 4 | 6 7 | 8 9 | 10 .. 13
    const unsigned long long first = 0xA8635210ULL;
    const int f = int((first >> (4 * warp)) & 15);
    const int cnt = warp < 4 ? 1 : (warp < 7 ? 2 : 4);
    return n < cnt ? f + n : -1;
  } else {
    // 0 | 1 | 2 | 3 4
    return n == 0 ? warp : (warp == 3 && n == 1 ? 4 : -1);
  }
}

// What an assembly reads besides the grid: T = double: the Gauss-point
// coefficients coef[(q NCF + k) NE + e]; T = float: the NN moments of the
// same coefficients mom[(k 3^D + w) NE + e], w = c_x 3^(D-1) + ..., with the
// powers of two sa, sb that derivatives on a coarse element carry.
template <class T>
struct AsmIn {
  const T* src;
  T lam, mu, kc;  // kc: w Gc l_s / h^2, times the unit products' scale
  T sa, sb;       // factors of A (both differentiated) and of B (one)
};

// The family moments of one element from the stored NN moments.
template <int D>
__device__ __forceinline__ void stored_family(const float* __restrict__ src, long long NE,
                                              long long e, bool in, int comp, float scale, int fam,
                                              int k, int l, float* out) {
  constexpr int E = Asm<D, float>::E, NW = Asm<D, float>::NW, W = 3 * NW;
  const float* s = src + (long long)comp * W * NE + e;
  int st[3] = {NW, D == 3 ? 3 : 1, 1};  // stride of c_x, c_y, c_z in w
  const int u = fam == 1 ? l : other(k, 0);
  const int v = D == 3 ? (fam == 1 ? 3 - k - l : other(k, 1)) : 0;
  // 32-bit offsets: 27 NE < 2^32 for any coarse level that fits the memory
  const unsigned ne = unsigned(NE);
  auto at = [&](int w) { return in ? scale * s[unsigned(w) * ne] : 0.f; };
  if (fam == 3) {
#pragma unroll
    for (int w = 0; w < W; ++w) out[w * E] = at(w);
    return;
  }
  const int sk = D == 3 ? (k == 0 ? st[0] : (k == 1 ? st[1] : st[2])) : (k == 0 ? st[0] : st[1]);
  const int su = D == 3 ? (u == 0 ? st[0] : (u == 1 ? st[1] : st[2])) : (u == 0 ? st[0] : st[1]);
  const int sv = D == 3 ? (v == 0 ? st[0] : (v == 1 ? st[1] : st[2])) : 0;
  constexpr int NV = D == 3 ? 3 : 1;
  if (fam == 1) {
    // N on k, N on u = l, NN on v
#pragma unroll
    for (int r = 0; r < NV; ++r) {
      float n[3][2];  // [c_u][beta]
#pragma unroll
      for (int p = 0; p < 3; ++p) {
        const float w0 = at(p * su + r * sv), w1 = at(sk + p * su + r * sv), w2 = at(2 * sk + p * su + r * sv);
        n[p][0] = w0 + w1;
        n[p][1] = w1 + w2;
      }
#pragma unroll
      for (int be = 0; be < 2; ++be)
#pragma unroll
        for (int al = 0; al < 2; ++al)
          out[((be * 2 + al) * NV + r) * E] = n[al][be] + n[al + 1][be];
    }
    return;
  }
#pragma unroll
  for (int p = 0; p < 3; ++p)
#pragma unroll
    for (int r = 0; r < NV; ++r) {
      const float w0 = at(p * su + r * sv), w1 = at(sk + p * su + r * sv), w2 = at(2 * sk + p * su + r * sv);
      const int idx = p * NV + r;
      if (fam == 0) {
        out[idx * E] = (w0 + w1) + (w1 + w2);
      } else {
        out[idx * E] = w0 + w1;
        out[(NW + idx) * E] = w1 + w2;
      }
    }
}

template <int D, class T>
__global__ void __launch_bounds__(Asm<D, T>::THREADS, Asm<D, T>::PER_SM)
    k_assemble(Geom g, AsmIn<T> in_, T* __restrict__ S, int tiles_x, int tiles_y, int chunk) {
  using A = Asm<D, T>;
  constexpr int F = A::F, E = A::E, FF = F * F;
  extern __shared__ double sm_raw[];
  T* mom = reinterpret_cast<T*>(sm_raw);  // [ROWS][E]
  T* carry = mom + A::ROWS * E;           // [CARRY][F F][32]
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  constexpr int MA = D - 1;  // march axis
  unsigned blk = blockIdx.x;
  const int ox = int(blk % unsigned(tiles_x)) * A::TX;
  blk /= unsigned(tiles_x);
  const int oy = D == 3 ? int(blk % unsigned(tiles_y)) * A::TY : 0;
  if (D == 3) blk /= unsigned(tiles_y);
  const int m0 = int(blk) * chunk, m1 = min(m0 + chunk, g.n[MA]);
  const PairConst<T> pc{in_.lam, -in_.lam, in_.mu, -in_.mu, in_.lam + T(2) * in_.mu,
                        -(in_.lam + T(2) * in_.mu)};
  const T* __restrict__ src = in_.src;
  const int nx = lane % A::TX, ny = lane / A::TX;
  const int gx = ox + nx, gy = oy + ny;
  for (int i = threadIdx.x; i < A::CARRY * FF * 32; i += A::THREADS) carry[i] = T(0);
  // element layer em lies between node layers em and em + 1
  for (int em = m0 - 1; em < m1; ++em) {
    __syncthreads();  // the previous layer's moments are read
    const bool layer = em >= 0 && em < g.ne[MA];
    for (int wt = warp; wt < A::W_ALL; wt += A::WARPS) {
      int t = wt, fam = 0;
      if (t >= A::W_DD) { t -= A::W_DD; fam = 1;
        if (t >= A::W_DN) { t -= A::W_DN; fam = 2;
          if (t >= A::W_BB) { t -= A::W_BB; fam = 3; } } }
      const int item = t * 32 + lane;
      const int e = item % E, mem = item / E;
      const int per = fam == 0 ? D : (fam == 1 ? A::PAIRS : (fam == 2 ? D * D : 1));
      if (mem >= per) continue;
      const int ex = ox - 1 + e % A::EX, ey = D == 3 ? oy - 1 + e / A::EX : em;
      const bool in = layer && ex >= 0 && ex < g.ne[0] && (D == 2 || (ey >= 0 && ey < g.ne[1]));
      const long long ge = D == 3 ? ex + (long long)g.ne[0] * (ey + (long long)g.ne[1] * em)
                                  : ex + (long long)g.ne[0] * em;
      // family member: its axes, its coefficient (A 0, M 1, B 2 + ...) and
      // where its moments go
      int k = mem, l = 0, comp = 0, base = A::DD + mem * A::NW;
      if (fam == 1) {
        k = D == 3 && mem == 2 ? 1 : 0;
        l = D == 3 && mem != 0 ? 2 : 1;
        base = A::DN + mem * A::NDN;
      } else if (fam == 2) {
        k = mem % D;
        comp = 2 + sym_index<D>(mem / D, k);
        base = A::BB + mem * 2 * A::NW;
      } else if (fam == 3) {
        comp = 1;
        base = A::MM;
        mom[A::COUNT * E + e] = in ? in_.kc : T(0);
      }
      T* out = mom + base * E + e;
      if constexpr (sizeof(T) == 4) {
        stored_family<D>(src, g.NE, ge, in, comp, fam < 2 ? in_.sa : (fam == 2 ? in_.sb : 1.f), fam,
                         k, l, out);
      } else {
        double v[(1 << D)];
        if (fam == 1)
          load_q<D>(src, g.NE, ge, in, comp, k, l, D == 3 ? 3 - k - l : 0, v);
        else if (fam == 3)
          load_q<D>(src, g.NE, ge, in, comp, 0, 1, 2, v);
        else
          load_q<D>(src, g.NE, ge, in, comp, k, other(k, 0), D == 3 ? other(k, 1) : 0, v);
        if (fam == 0) moments_dd<D>(v, out);
        else if (fam == 1) moments_dn<D>(v, out);
        else if (fam == 2) moments_b<D>(v, out);
        else moments_m<D>(v, out);
      }
    }
    __syncthreads();
#pragma unroll 1
    for (int n = 0;; ++n) {
      const int j = warp_offset<D>(warp, n);
      if (j < 0) break;
      int o[3];
      half_offset<D>(j, o);
      // the pairs of node layer em (corner 0 along the march axis), then,
      // for blocks along no march axis, those of node layer em + 1
      const int sides = o[MA] == 0 ? 2 : 1;
      T tot[FF];
#pragma unroll
      for (int i = 0; i < FF; ++i) tot[i] = j < A::CARRY ? carry[(j * FF + i) * 32 + lane] : T(0);
#pragma unroll 1
      for (int side = 0; side < sides; ++side) {
        if (side == 0 && em < m0) continue;
        if (side == 1) {
          if (em == m1 - 1) break;  // the next chunk's nodes
#pragma unroll
          for (int i = 0; i < FF; ++i) tot[i] = T(0);
        }
#pragma unroll 1
        for (int q = 0; q < (1 << MA); ++q) {  // corner of the node off the march axis
          const int a0 = q & 1, a1 = D == 3 ? q >> 1 : side, a2 = D == 3 ? side : 0;
          const int b0 = a0 + o[0], b1 = a1 + o[1], b2 = a2 + o[2];
          if (b0 < 0 || b0 > 1 || b1 < 0 || b1 > 1 || b2 < 0 || b2 > 1) continue;
          const int el = (nx - a0 + 1) + (D == 3 ? A::EX * (ny - a1 + 1) : 0);
          add_pair<D, T>(mom + el, a0 | a1 << 1 | a2 << 2, b0 | b1 << 1 | b2 << 2, pc, tot);
        }
        if (side == 0) {
          const int gz = D == 3 ? em : 0, y = D == 3 ? gy : em;
          if (gx < g.n[0] && y < g.n[1]) {
            const long long i = gx + g.n[0] * (y + (long long)g.n[1] * gz);
            auto inside = [&](int s) {
              const int x = gx + s * o[0], yy = y + s * o[1], z = gz + s * o[2];
              return x >= 0 && x < g.n[0] && yy >= 0 && yy < g.n[1] && z >= 0 && z < g.n[2];
            };
            const long long shift = o[0] + g.n[0] * (o[1] + (long long)g.n[1] * o[2]);
            const int code = (o[0] + 1) + 3 * (o[1] + 1) + (D == 3 ? 9 * (o[2] + 1) : 0);
            const int opp = (D == 3 ? 26 : 8) - code;
            const bool fwd = inside(1), back = inside(-1);
            // entry (f, h) of block o, then entry (h, f) of block -o: plane
            // by plane with a running pointer
            T* p = S + (long long)code * FF * g.N + i;
#pragma unroll
            for (int k = 0; k < FF; ++k, p += g.N) *p = fwd ? tot[k] : T(0);
            if (j > 0) {
              p = S + (long long)opp * FF * g.N + i;
              if (!back) {
                T* z = p;
#pragma unroll
                for (int k = 0; k < FF; ++k, z += g.N) *z = T(0);
              }
              if (fwd) {
                p += shift;
#pragma unroll
                for (int k = 0; k < FF; ++k, p += g.N) *p = tot[(k % F) * F + k / F];
              }
            }
          }
        }
      }
      if (sides == 2)
#pragma unroll
        for (int i = 0; i < FF; ++i) carry[(j * FF + i) * 32 + lane] = tot[i];
    }
  }
}

template <int D, class T>
cudaError_t launch(const Geom& g, const AsmIn<T>& in, T* S, cudaStream_t st) {
  using A = Asm<D, T>;
  cudaError_t e = cudaFuncSetAttribute(k_assemble<D, T>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       int(A::smem));
  if (e != cudaSuccess) return e;
  const int tx = (g.n[0] + A::TX - 1) / A::TX, ty = D == 3 ? (g.n[1] + A::TY - 1) / A::TY : 1;
  const int nm = g.n[D - 1];
  // Chunks of node layers: a chunk forms one element layer more than it has
  // nodes (about 0.7 of a layer's work), and the CTAs run in waves of PER_SM
  // per SM.  Take the count with the least layers x waves.
  const long long tiles = (long long)tx * ty, slots = A::PER_SM * 152;
  int chunk = nm;
  double best = 1e300;
  for (int c = 1; c <= std::min(nm, 512); ++c) {
    const int len = (nm + c - 1) / c;
    const double waves = double((tiles * ((nm + len - 1) / len) + slots - 1) / slots);
    if (waves * (len + 0.7) < best) {
      best = waves * (len + 0.7);
      chunk = len;
    }
  }
  const long long blocks = tiles * ((nm + chunk - 1) / chunk);
  if (blocks > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
  k_assemble<D, T><<<unsigned(blocks), A::THREADS, A::smem, st>>>(g, in, S, tx, ty, chunk);
  return cudaGetLastError();
}

}  // namespace

cudaError_t stencil_assemble(const Geom& g, const Mat<double>& m, const double* coef, double* S,
                             cudaStream_t st) {
  const AsmIn<double> in{coef, m.lam, m.mu, m.w * m.Gc * m.ls * m.inv_h * m.inv_h, 1.0, 1.0};
  return g.dim == 3 ? launch<3, double>(g, in, S, st) : launch<2, double>(g, in, S, st);
}

cudaError_t galerkin_assemble(const Geom& g, const Mat<double>& mf, int depth, const float* mom,
                              float* S, cudaStream_t st) {
  // a derivative on an element 2^depth times as wide is 2^-depth of one on a
  // fine element; of a constant coefficient's products per axis, "both
  // differentiated" sums to 2^-depth and NN to 2^depth of the fine element's
  const double s = std::ldexp(1.0, -depth);
  const double kc = mf.w * mf.Gc * mf.ls * mf.inv_h * mf.inv_h * std::ldexp(1.0, (g.dim - 2) * depth);
  const AsmIn<float> in{mom, float(mf.lam), float(mf.mu), float(kc), float(s * s), float(s)};
  return g.dim == 3 ? launch<3, float>(g, in, S, st) : launch<2, float>(g, in, S, st);
}

}  // namespace pf
