// Learned initial iterate: a 2D U-Net (4 levels, two 3x3 convolutions +
// ReLU per level, 2x2 average pooling down, nearest 2x up, skip
// concatenation, 1x1 head).  BF16 weights and activations, FP32 master
// weights and Adam moments.  Every convolution (forward, data gradient,
// weight gradient) is an implicit GEMM on the tensor cores with BF16
// operands and FP32 accumulation; the data-gradient and weight-gradient
// operand dL/d(out) (FP32) is split into a BF16 pair hi + lo and multiplied
// twice, keeping about 16 significant bits of the gradient.
//
// Layout.  Activations are channel-innermost ([y][x][channel], channels
// padded to 16 with zeros), so that 16 channels of a pixel are two 16-byte
// cp.async pieces and an ldmatrix row is 8 channels of any pixel: a tap is a
// shift of row addresses.  With channel planes every operand word was two
// scalar loads with the pooling, upsampling or concatenation worked out per
// value, and the tensor pipe was 4-9 % busy; now it is 34-70 % busy (of what
// mma.sync can issue) in the 3 x 3 products of 1032^2, but for those whose
// epilogue spreads a pooled gradient (15-19 %), and 6-11 % in the 1 x 1 head.  Forward and backward:
//   1032^2  1.92 -> 0.44 ms and  9.19 -> 1.61 ms
//    136^2   604 ->   66 us and  1183 ->  271 us (latency of 16 and 45
//                                                launches in sequence)
// The input transforms need no passes of their own:
//  - the second convolution of an encoder level also writes the 2x2 average
//    the next level reads (a thread holds both rows of a pixel pair);
//  - nearest upsampling and the skip concatenation are source addresses.
// The backward pass stores no FP32 gradient but those of the skips: a data
// gradient's epilogue applies the adjoint of the input transform in FP32
// (with the skip's gradient where there is one), masks by the ReLU of the
// layer below, adds that layer's bias gradient and writes the hi + lo pair
// the next two products read.
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <string>
#include <vector>

#include "../../include/pf.h"
#include "pf_internal.h"

namespace pf {
void set_error(const std::string& msg);
}
using namespace pf;

namespace {

typedef __nv_bfloat16 bf16;
typedef __nv_bfloat162 bf162;

// Input of a convolution on an H x W grid: channels [0, ca) from a (at half
// the resolution with up), then [ca, ca + cb) from b; both padded to 16.
struct ConvSrc {
  const bf16* a;
  int ca, up;
  const bf16* b;
  int cb;
};

// ---------------------------------------------------------------- primitives
__device__ __forceinline__ unsigned smem_addr(const void* p) {
  return unsigned(__cvta_generic_to_shared(p));
}
// 16 bytes to shared memory, zeros where !in
__device__ __forceinline__ void cp16(unsigned dst, const void* src, bool in) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(in ? 16 : 0));
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;"); }
template <int N>
__device__ __forceinline__ void cp_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N));
}
__device__ __forceinline__ void ldm4(unsigned (&r)[4], unsigned a) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(a));
}
__device__ __forceinline__ void ldm4t(unsigned (&r)[4], unsigned a) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(a));
}
__device__ __forceinline__ void ldm2t(unsigned (&r)[2], unsigned a) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x2.trans.shared.b16 {%0,%1}, [%2];"
               : "=r"(r[0]), "=r"(r[1]) : "r"(a));
}
// one warp-wide 16 x 8 x 16 product
__device__ __forceinline__ void mma_bf16(float (&c)[4], const unsigned (&a)[4], unsigned b0,
                                         unsigned b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, "
      "{%8,%9}, {%0,%1,%2,%3};\n"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// Byte offset of 16-byte piece c of row p in a tile of rows of CH channels;
// the pieces are permuted so that eight consecutive rows' pieces c fall in
// distinct banks.
template <int CH>
__device__ __forceinline__ int swz(int p, int c) {
  static_assert(CH == 16 || CH == 32, "rows of 16 or 32 channels");
  return CH == 16 ? p * 32 + ((c ^ ((p >> 2) & 1)) << 4) : p * 64 + ((c ^ ((p >> 1) & 3)) << 4);
}

// v = hi + lo, both BF16 (about 16 significant bits)
__device__ __forceinline__ void split2(float v0, float v1, bf162& hi, bf162& lo) {
  hi = __floats2bfloat162_rn(v0, v1);
  lo = __floats2bfloat162_rn(v0 - __low2float(hi), v1 - __high2float(hi));
}

// ---------------------------------------------------------------- convolution
// Forward:  out[p][co]  = sum_{ci, tap} in[p + off(tap)][ci] w[co][ci][tap]
// Data gradient: din[p][ci] = sum_{co, tap} dpre[p + off(tap)][co] w[co][ci][KK-1-tap]
// Both are M = pixels, N = output channels, K = input channels of each tap.
// A CTA takes 16 x 8 pixels and NB output channels; a warp takes XT = 1 or 2
// M tiles of 2 x 8 pixels (side by side in two pixel rows) and all NB
// channels, so there are 8 or 4 warps.  Input
// channels come in chunks of 16, staged with their weights by cp.async in a
// ring of ST stages; per chunk the taps run in order, so an output's sum is
// over (chunk, tap) in a fixed order whatever NB is.
enum { EPI_FWD = 0, EPI_HEAD = 1, EPI_PLAIN = 2, EPI_POOL = 3, EPI_UP = 4 };

struct EpiArgs {
  const float* bias;   // EPI_FWD, EPI_HEAD
  int co;              // real output channels (EPI_FWD, EPI_HEAD)
  int cp;              // padded channels of the tensor written
  bf16* out;           // EPI_FWD: activation
  bf16* pool;          // EPI_FWD: its 2 x 2 average, or null
  float* y;            // EPI_HEAD: planes
  // gradient of the layer below (activation act, cp channels): hi + lo pair
  const bf16* act;
  bf16 *hi, *lo;
  const float* skip_in;  // EPI_POOL: gradient through the skip, FP32, on act's grid
  float* skip_out;       // EPI_UP: gradient of the concatenated skip (cb channels)
  int ca, cb;            // EPI_UP: channels of the upsampled operand and of the skip
  float* part_b;         // bias gradient of the layer below: [tile][cp]
};

constexpr int TW = 16, TH = 8;  // pixels of a CTA

template <int K, int NB, int NS>
struct ConvSmem {
  static constexpr int R = K / 2, XW = TW + 2 * R, XH = TH + 2 * R, NP = XW * XH, KK = K * K;
  static constexpr int px = NS * NP * 32, stage = px + KK * NB * 32;
  // stages: up to eight within 84 KB; a launch takes no more than it has chunks
  static constexpr int FIT = 84 * 1024 / stage, ST = FIT > 8 ? 8 : FIT;
  static constexpr int bytes = ST * stage;
};

template <int K, int NB, int XT, int EPI>
__global__ void __launch_bounds__(256 / XT)
    k_conv(ConvSrc s, const bf16* __restrict__ s_lo, const bf16* __restrict__ w, int H, int W, int KC,
           EpiArgs e) {
  constexpr bool GRAD = EPI >= EPI_PLAIN;
  constexpr int NS = GRAD ? 2 : 1;
  using S = ConvSmem<K, NB, NS>;
  constexpr int R = S::R, XW = S::XW, NP = S::NP, KK = S::KK, ST = S::ST, NT = NB / 8;
  constexpr int THREADS = 256 / XT, WARPS = 8 / XT;
  extern __shared__ __align__(16) unsigned char smem[];
  const unsigned sm = smem_addr(smem);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int rows = 2 * (XT == 2 ? warp : warp >> 1), xw = XT == 2 ? 0 : (warp & 1) * 8;  // the warp's pixels
  const int g = lane >> 2, t4 = lane & 3;
  const int x0 = blockIdx.x * TW, y0 = blockIdx.y * TH, n0 = blockIdx.z * NB;

  auto load_weights = [&](int kc, int buf) {
    // [group of 16 outputs][chunk][tap][16 outputs][16 inputs]
    const unsigned d = sm + buf * S::stage + S::px;
    for (int i = threadIdx.x; i < KK * NB * 2; i += THREADS) {
      const int h = i & 1, n = (i >> 1) & 15, r = i >> 5, tap = r % KK, cg = r / KK;
      const long long o = ((((long long)(n0 / 16 + cg) * KC + kc) * KK + tap) * 16 + n) * 16 + h * 8;
      cp16(d + swz<16>(tap * NB + cg * 16 + n, h), w + o, true);
    }
  };
  auto load_pixels = [&](int kc, int buf) {
    const unsigned d = sm + buf * S::stage;
    const int c0 = kc * 16;
    const bool from_a = GRAD || c0 < s.ca;
    const bf16* src = from_a ? s.a : s.b;
    const int cs = from_a ? s.ca : s.cb, co = from_a ? c0 : c0 - s.ca;
    const int sh = from_a && s.up ? 1 : 0, ws = W >> sh;
    for (int i = threadIdx.x; i < NP * 2; i += THREADS) {
      const int p = i >> 1, h = i & 1;
      const int yy = y0 - R + p / XW, xx = x0 - R + p % XW;
      const bool in = yy >= 0 && yy < H && xx >= 0 && xx < W;
      const long long o = in ? ((long long)(yy >> sh) * ws + (xx >> sh)) * cs + co + h * 8 : 0;
      cp16(d + swz<16>(p, h), src + o, in);
      if constexpr (NS == 2) cp16(d + NP * 32 + swz<16>(p, h), s_lo + o, in);
    }
  };

  float acc[XT][NT][4];
#pragma unroll
  for (int a = 0; a < XT; ++a)
#pragma unroll
    for (int b = 0; b < NT; ++b)
#pragma unroll
      for (int c = 0; c < 4; ++c) acc[a][b][c] = 0.f;

  // the weights do not depend on the launch before (only on one further back):
  // fetch the first of them while it finishes, then let the next launch start
#pragma unroll
  for (int st = 0; st < ST - 1; ++st)
    if (st < KC) load_weights(st, st);
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;");
#pragma unroll
  for (int st = 0; st < ST - 1; ++st) {
    if (st < KC) load_pixels(st, st);
    cp_commit();
  }
  // ldmatrix rows of this lane: A row (pixel) and half, B row (channel) and half
  const int a_q = (rows + ((lane >> 3) & 1)) * XW + xw + (lane & 7), a_h = lane >> 4;
  const int b_n = (lane & 7) + 8 * (lane >> 4), b_h = (lane >> 3) & 1;
  for (int kc = 0; kc < KC; ++kc) {
    cp_wait<ST - 2>();
    __syncthreads();
    if (kc + ST - 1 < KC) {
      load_weights(kc + ST - 1, (kc + ST - 1) % ST);
      load_pixels(kc + ST - 1, (kc + ST - 1) % ST);
    }
    cp_commit();
    const unsigned px = sm + (kc % ST) * S::stage, wt = px + S::px;
#pragma unroll
    for (int tap = 0; tap < KK; ++tap) {
      const int ky = tap / K, kx = tap % K;
      unsigned a[NS][XT][4], b[NT / 2][4];
#pragma unroll
      for (int part = 0; part < NS; ++part)
#pragma unroll
        for (int xt = 0; xt < XT; ++xt)
          ldm4(a[part][xt], px + part * NP * 32 + swz<16>(a_q + ky * XW + kx + xt * 8, a_h));
#pragma unroll
      for (int j = 0; j < NT / 2; ++j) ldm4(b[j], wt + swz<16>(tap * NB + j * 16 + b_n, b_h));
#pragma unroll
      for (int part = 0; part < NS; ++part)
#pragma unroll
        for (int xt = 0; xt < XT; ++xt)
#pragma unroll
          for (int nt = 0; nt < NT; ++nt)
            mma_bf16(acc[xt][nt], a[part][xt], b[nt / 2][(nt & 1) * 2], b[nt / 2][(nt & 1) * 2 + 1]);
    }
  }
  cp_wait<0>();

  // epilogue: lane (g, t4) holds pixels (y, x), (y + 1, x) of channels ch, ch + 1
  const int y = y0 + rows;
  float bsum[NT][2];
#pragma unroll
  for (int nt = 0; nt < NT; ++nt) bsum[nt][0] = bsum[nt][1] = 0.f;
  // gradient of the layer below at pixel o (of its grid): mask, split, bias
  auto grad_out = [&](long long o, int ch, float v0, float v1, float (&bs)[2]) {
    const long long k = o * e.cp + ch;
    const bf162 a = *reinterpret_cast<const bf162*>(e.act + k);
    v0 = __low2float(a) > 0.f ? v0 : 0.f;
    v1 = __high2float(a) > 0.f ? v1 : 0.f;
    bf162 hi, lo;
    split2(v0, v1, hi, lo);
    *reinterpret_cast<bf162*>(e.hi + k) = hi;
    *reinterpret_cast<bf162*>(e.lo + k) = lo;
    bs[0] += v0;
    bs[1] += v1;
  };
#pragma unroll
  for (int xt = 0; xt < XT; ++xt) {
    const int x = x0 + xw + xt * 8 + g;
#pragma unroll
    for (int nt = 0; nt < NT; ++nt) {
      const int ch = n0 + nt * 8 + 2 * t4;
      float(&c)[4] = acc[xt][nt];
      const bool in0 = x < W && y < H, in1 = x < W && y + 1 < H;
      if constexpr (EPI == EPI_FWD || EPI == EPI_HEAD) {
        const float b0 = ch < e.co ? e.bias[ch] : 0.f, b1 = ch + 1 < e.co ? e.bias[ch + 1] : 0.f;
        if constexpr (EPI == EPI_HEAD) {
          const long long HW = (long long)H * W, o = (long long)y * W + x;
          if (ch < e.co) {
            if (in0) e.y[ch * HW + o] = c[0] + b0;
            if (in1) e.y[ch * HW + o + W] = c[2] + b0;
          }
          if (ch + 1 < e.co) {
            if (in0) e.y[(ch + 1) * HW + o] = c[1] + b1;
            if (in1) e.y[(ch + 1) * HW + o + W] = c[3] + b1;
          }
        } else {
          const bf162 r0 = __floats2bfloat162_rn(fmaxf(c[0] + b0, 0.f), fmaxf(c[1] + b1, 0.f));
          const bf162 r1 = __floats2bfloat162_rn(fmaxf(c[2] + b0, 0.f), fmaxf(c[3] + b1, 0.f));
          bf16* o = e.out + ((long long)y * W + x) * e.cp + ch;
          if (ch < e.cp) {
            if (in0) *reinterpret_cast<bf162*>(o) = r0;
            if (in1) *reinterpret_cast<bf162*>(o + (long long)W * e.cp) = r1;
          }
          if (e.pool) {
            // the average of the stored (rounded) values, ((00 + 01) + 10) + 11
            const float p0 = __low2float(r0), p1 = __high2float(r0);
            const float q0 = __low2float(r1), q1 = __high2float(r1);
            const float pr0 = __shfl_xor_sync(0xffffffffu, p0, 4), pr1 = __shfl_xor_sync(0xffffffffu, p1, 4);
            const float qr0 = __shfl_xor_sync(0xffffffffu, q0, 4), qr1 = __shfl_xor_sync(0xffffffffu, q1, 4);
            if (!(g & 1) && in1 && ch < e.cp)
              *reinterpret_cast<bf162*>(e.pool + ((long long)(y >> 1) * (W >> 1) + (x >> 1)) * e.cp + ch) =
                  __floats2bfloat162_rn(0.25f * (p0 + pr0 + q0 + qr0), 0.25f * (p1 + pr1 + q1 + qr1));
          }
        }
      } else if constexpr (EPI == EPI_PLAIN) {
        if (ch < e.cp) {
          if (in0) grad_out((long long)y * W + x, ch, c[0], c[1], bsum[nt]);
          if (in1) grad_out((long long)(y + 1) * W + x, ch, c[2], c[3], bsum[nt]);
        }
      } else if constexpr (EPI == EPI_POOL) {
        // each coarse value goes to its 2 x 2 pixels with weight 1/4
        if (ch < e.cp) {
          const int W2 = 2 * W;
#pragma unroll
          for (int r = 0; r < 2; ++r) {
            if (!(r ? in1 : in0)) continue;
            const float v0 = 0.25f * c[2 * r], v1 = 0.25f * c[2 * r + 1];
#pragma unroll
            for (int d = 0; d < 4; ++d) {
              const long long o = (long long)(2 * (y + r) + (d >> 1)) * W2 + 2 * x + (d & 1);
              const float2 sk = *reinterpret_cast<const float2*>(e.skip_in + o * e.cp + ch);
              grad_out(o, ch, sk.x + v0, sk.y + v1, bsum[nt]);
            }
          }
        }
      } else {
        if (n0 + nt * 8 < e.ca) {
          // the upsampled operand: sums of 2 x 2 pixels, ((00 + 01) + 10) + 11
          const float r0 = __shfl_xor_sync(0xffffffffu, c[0], 4), r1 = __shfl_xor_sync(0xffffffffu, c[1], 4);
          const float r2 = __shfl_xor_sync(0xffffffffu, c[2], 4), r3 = __shfl_xor_sync(0xffffffffu, c[3], 4);
          if (!(g & 1) && in1)
            grad_out((long long)(y >> 1) * (W >> 1) + (x >> 1), ch, c[0] + r0 + c[2] + r2,
                     c[1] + r1 + c[3] + r3, bsum[nt]);
        } else if (ch < e.ca + e.cb) {
          float* o = e.skip_out + ((long long)y * W + x) * e.cb + ch - e.ca;
          if (in0) *reinterpret_cast<float2*>(o) = make_float2(c[0], c[1]);
          if (in1) *reinterpret_cast<float2*>(o + (long long)W * e.cb) = make_float2(c[2], c[3]);
        }
      }
    }
  }
  if constexpr (GRAD) {
    // bias gradient of the layer below: lanes of a channel, then warps
    __syncthreads();
    float* sb = reinterpret_cast<float*>(smem);  // [warp][NB]
#pragma unroll
    for (int nt = 0; nt < NT; ++nt)
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        float v = bsum[nt][k];
        v += __shfl_xor_sync(0xffffffffu, v, 4);
        v += __shfl_xor_sync(0xffffffffu, v, 8);
        v += __shfl_xor_sync(0xffffffffu, v, 16);
        if (g == 0) sb[warp * NB + nt * 8 + 2 * t4 + k] = v;
      }
    __syncthreads();
    const int ch = n0 + threadIdx.x;
    if (threadIdx.x < NB && ch < e.cp) {
      float t = 0.f;
#pragma unroll
      for (int r = 0; r < WARPS; ++r) t += sb[r * NB + threadIdx.x];
      e.part_b[((long long)blockIdx.y * gridDim.x + blockIdx.x) * e.cp + ch] = t;
    }
  }
}

// Opt-in to dynamic shared memory above 48 KB, once per kernel, device and
// thread.
template <class F>
cudaError_t opt_in(F kernel, int bytes, int& done_dev) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess || done_dev == dev) return e;
  e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  if (e == cudaSuccess) done_dev = dev;
  return e;
}

template <int K, int NB, int XT, int EPI>
cudaError_t launch_conv_nb(const ConvSrc& s, const bf16* lo, const bf16* w, int H, int W, int N, int KC,
                           const EpiArgs& e, cudaStream_t st) {
  using S = ConvSmem<K, NB, (EPI >= EPI_PLAIN ? 2 : 1)>;
  static thread_local int done = -1;
  cudaError_t rc = opt_in(k_conv<K, NB, XT, EPI>, S::bytes, done);
  if (rc != cudaSuccess) return rc;
  // programmatic dependent launch: the CTAs start while the launch before
  // drains and wait for it where they first read what it wrote
  cudaLaunchAttribute attr{};
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((W + TW - 1) / TW, (H + TH - 1) / TH, N / NB);
  cfg.blockDim = dim3(256 / XT);
  cfg.dynamicSmemBytes = size_t(std::min(S::ST, KC)) * S::stage;
  cfg.stream = st;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k_conv<K, NB, XT, EPI>, s, lo, w, H, W, KC, e);
}

// N output channels (a multiple of 16) in blocks of 64, 32 or 16: the largest
// that divides N and leaves two CTAs per SM.  A block of 64 reuses a pixel
// fragment eight times where 16 reuses it twice, but the deep levels have few
// pixel tiles (at 136^2 and 17 x 17 pixels: 6) and there the parallelism wins;
// a launch below two CTAs per SM also halves each warp's share (8 warps with
// one M tile: its length is then set by one warp's instruction latencies).
template <int K, int EPI>
cudaError_t launch_conv(const ConvSrc& s, const bf16* lo, const bf16* w, int H, int W, int N, int KC,
                        const EpiArgs& e, int sms, cudaStream_t st) {
  const long long tiles = (long long)((W + TW - 1) / TW) * ((H + TH - 1) / TH);
  const auto full = [&](int nb) { return N % nb == 0 && tiles * (N / nb) >= 2LL * sms; };
  if (full(64)) return launch_conv_nb<K, 64, 2, EPI>(s, lo, w, H, W, N, KC, e, st);
  if (full(32)) return launch_conv_nb<K, 32, 2, EPI>(s, lo, w, H, W, N, KC, e, st);
  if (full(16)) return launch_conv_nb<K, 16, 2, EPI>(s, lo, w, H, W, N, KC, e, st);
  return launch_conv_nb<K, 16, 1, EPI>(s, lo, w, H, W, N, KC, e, st);
}

// ---------------------------------------------------------------- weight gradient
// dw[co][ci][tap] = sum_p dpre[p][co] in[p + off(tap)][ci]: M = co, N = ci,
// K = pixels, 16 of a tile row at a time.  Both operands are channel-innermost
// tiles, so their fragments are transposing ldmatrix reads.  A CTA of 8 warps
// takes MB x NB channels and a contiguous chunk of the layer's 16 x 16 pixel
// tiles (staged in two alternating buffers by cp.async); a warp takes one
// 16 x 8 block of (co, ci) with all its taps, marching down rows with the
// input fragments of three rows in registers: a row's six loads (2 of dpre,
// 3 of the input) feed 18 products.  Where MB x NB has fewer than 8 blocks
// the warps share the rows and their sums are added at the end.
template <int K, int MB, int NB>
struct WgradSmem {
  static constexpr int R = K / 2, XW = 16 + 2 * R, NX = XW * XW, KK = K * K;
  static constexpr int BLK = (MB / 16) * (NB / 8), KG = 8 / BLK, ROWS = 16 / KG;
  static constexpr int d_part = 256 * MB * 2, x_off = 2 * d_part, stage = x_off + NX * NB * 2;
  static constexpr int red = 8 * KK * 4 * 32 * 4;
  static constexpr int bytes = 2 * stage > red ? 2 * stage : red;
};

template <int K, int MB, int NB>
__global__ void __launch_bounds__(256, 2)
    k_wgrad(const bf16* __restrict__ dh, const bf16* __restrict__ dl, int coP, ConvSrc in, int ca,
            int cb, int H, int W, int CO, int P, float* __restrict__ part) {
  using S = WgradSmem<K, MB, NB>;
  constexpr int R = S::R, XW = S::XW, KK = S::KK, KG = S::KG, ROWS = S::ROWS;
  extern __shared__ __align__(16) unsigned char smem[];
  const unsigned sm = smem_addr(smem);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int blk = warp % S::BLK, kg = warp / S::BLK;
  const int mt = blk % (MB / 16), nt = blk / (MB / 16);
  const int n0 = blockIdx.x * NB, m0 = blockIdx.y * MB, p = blockIdx.z;
  const int tx = (W + 15) / 16;
  const long long T = (long long)tx * ((H + 15) / 16);
  const long long t_lo = p * T / P, t_hi = (p + 1) * T / P;

  auto load = [&](long long ti, int buf) {
    const unsigned d = sm + buf * S::stage;
    const int yb = int(ti / tx) * 16, xb = int(ti % tx) * 16;
    for (int i = threadIdx.x; i < 256 * (MB / 8); i += 256) {
      const int c = i % (MB / 8), q = i / (MB / 8);
      const int yy = yb + q / 16, xx = xb + q % 16, ch = m0 + c * 8;
      const bool ok = yy < H && xx < W && ch < coP;
      const long long o = ok ? ((long long)yy * W + xx) * coP + ch : 0;
      cp16(d + swz<MB>(q, c), dh + o, ok);
      cp16(d + S::d_part + swz<MB>(q, c), dl + o, ok);
    }
    for (int i = threadIdx.x; i < S::NX * (NB / 8); i += 256) {
      const int c = i % (NB / 8), q = i / (NB / 8);
      const int yy = yb - R + q / XW, xx = xb - R + q % XW, ch = n0 + c * 8;
      const bool a = ch < in.ca;
      const bool ok = yy >= 0 && yy < H && xx >= 0 && xx < W && ch < in.ca + in.cb;
      const int sh = a && in.up ? 1 : 0;
      const long long o = ok ? ((long long)(yy >> sh) * (W >> sh) + (xx >> sh)) * (a ? in.ca : in.cb) +
                                   (a ? ch : ch - in.ca)
                             : 0;
      cp16(d + S::x_off + swz<NB>(q, c), (a || !ok ? in.a : in.b) + o, ok);
    }
  };

  float acc[KK][4];
#pragma unroll
  for (int k = 0; k < KK; ++k)
#pragma unroll
    for (int c = 0; c < 4; ++c) acc[k][c] = 0.f;
  // transposed ldmatrix rows of this lane
  const int d_q = (lane >> 4) * 8 + (lane & 7), d_c = mt * 2 + ((lane >> 3) & 1);
  const int x_q = ((lane >> 3) & 1) * 8 + (lane & 7);
  if (t_lo < t_hi) load(t_lo, 0);
  cp_commit();
  for (long long ti = t_lo; ti < t_hi; ++ti) {
    const int buf = int((ti - t_lo) & 1);
    if (ti + 1 < t_hi) load(ti + 1, buf ^ 1);
    cp_commit();
    cp_wait<1>();
    __syncthreads();
    const unsigned d = sm + buf * S::stage, x = d + S::x_off;
    const int r0 = kg * ROWS;
    unsigned bf[K][K][2];  // [input row mod K][kx]
#pragma unroll
    for (int r = 0; r < K - 1; ++r)
#pragma unroll
      for (int kx = 0; kx < K; ++kx) ldm2t(bf[r][kx], x + swz<NB>((r0 + r) * XW + kx + x_q, nt));
#pragma unroll
    for (int r = 0; r < ROWS; ++r) {
      unsigned ah[4], al[4];
      ldm4t(ah, d + swz<MB>((r0 + r) * 16 + d_q, d_c));
      ldm4t(al, d + S::d_part + swz<MB>((r0 + r) * 16 + d_q, d_c));
#pragma unroll
      for (int kx = 0; kx < K; ++kx)
        ldm2t(bf[(r + K - 1) % K][kx], x + swz<NB>((r0 + r + K - 1) * XW + kx + x_q, nt));
#pragma unroll
      for (int tap = 0; tap < KK; ++tap) {
        const unsigned(&b)[2] = bf[(r + tap / K) % K][tap % K];
        mma_bf16(acc[tap], ah, b[0], b[1]);
        mma_bf16(acc[tap], al, b[0], b[1]);
      }
    }
    __syncthreads();
  }
  cp_wait<0>();
  if constexpr (KG > 1) {
    float* red = reinterpret_cast<float*>(smem);  // [warp][tap][4][lane]
    __syncthreads();
    if (kg > 0)
#pragma unroll
      for (int k = 0; k < KK; ++k)
#pragma unroll
        for (int c = 0; c < 4; ++c) red[((warp * KK + k) * 4 + c) * 32 + lane] = acc[k][c];
    __syncthreads();
    if (kg > 0) return;
#pragma unroll
    for (int o = 1; o < KG; ++o)
#pragma unroll
      for (int k = 0; k < KK; ++k)
#pragma unroll
        for (int c = 0; c < 4; ++c) acc[k][c] += red[(((warp + o * S::BLK) * KK + k) * 4 + c) * 32 + lane];
  }
  const int g = lane >> 2, t4 = lane & 3, CI = ca + cb;
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    const int co = m0 + mt * 16 + g + 8 * (c >> 1), cp = n0 + nt * 8 + 2 * t4 + (c & 1);
    // padded input channel -> real one
    const int ci = cp < in.ca ? (cp < ca ? cp : -1) : (cp - in.ca < cb ? ca + cp - in.ca : -1);
    if (co < CO && ci >= 0)
#pragma unroll
      for (int k = 0; k < KK; ++k) part[(((long long)p * CO + co) * CI + ci) * KK + k] = acc[k][c];
  }
}

// Channel blocks of a weight gradient: 32 where the layer has more than 16.
int wg_block(int cp) { return cp > 16 ? 32 : 16; }

// Pixel-tile chunks of a weight-gradient launch: enough for two CTAs per SM
// over the (input block, output block) grid, at most one chunk per tile.
int wgrad_chunks(int H, int W, int ciP, int coP, int sms) {
  const long long T = (long long)((W + 15) / 16) * ((H + 15) / 16);
  const int mb = wg_block(coP), nb = wg_block(ciP);
  const long long base = (long long)((ciP + nb - 1) / nb) * ((coP + mb - 1) / mb);
  const long long want = (2LL * sms + base - 1) / base;
  return int(std::max<long long>(1, std::min(T, want)));
}

template <int K, int MB, int NB>
cudaError_t launch_wgrad_b(const bf16* dh, const bf16* dl, int coP, const ConvSrc& in, int ca, int cb,
                           int H, int W, int CO, int P, float* part, cudaStream_t st) {
  using S = WgradSmem<K, MB, NB>;
  static thread_local int done = -1;
  cudaError_t rc = opt_in(k_wgrad<K, MB, NB>, S::bytes, done);
  if (rc != cudaSuccess) return rc;
  const dim3 grid((in.ca + in.cb + NB - 1) / NB, (coP + MB - 1) / MB, P);
  k_wgrad<K, MB, NB><<<grid, 256, S::bytes, st>>>(dh, dl, coP, in, ca, cb, H, W, CO, P, part);
  return cudaGetLastError();
}

template <int K>
cudaError_t launch_wgrad(const bf16* dh, const bf16* dl, int coP, const ConvSrc& in, int ca, int cb,
                         int H, int W, int CO, int P, float* part, cudaStream_t st) {
  const bool m32 = wg_block(coP) == 32, n32 = wg_block(in.ca + in.cb) == 32;
  if (m32 && n32) return launch_wgrad_b<K, 32, 32>(dh, dl, coP, in, ca, cb, H, W, CO, P, part, st);
  if (m32) return launch_wgrad_b<K, 32, 16>(dh, dl, coP, in, ca, cb, H, W, CO, P, part, st);
  if (n32) return launch_wgrad_b<K, 16, 32>(dh, dl, coP, in, ca, cb, H, W, CO, P, part, st);
  return launch_wgrad_b<K, 16, 16>(dh, dl, coP, in, ca, cb, H, W, CO, P, part, st);
}

// grad += sum_p part[p] for a layer's weights (n values, P partials) and
// biases (nb of the ldb columns, Pb partials).  A warp covers `cols`
// neighbouring values and 32 / cols partials at a time: few values with many
// partials (16 biases, 2,178 tiles at 528 x 520: 44 us with one value per
// lane) take narrow blocks.  Added in a fixed order: every (256 / cols)-th
// partial per thread, then a tree over the threads of a value.
__device__ __forceinline__ void sum_columns(const float* __restrict__ src, int P, long long n,
                                            long long ld, int cols, long long block,
                                            float* __restrict__ grad) {
  __shared__ float sh[256];
  const int col = threadIdx.x % cols, row = threadIdx.x / cols, rows = 256 / cols;
  const long long i = block * cols + col;
  float s = 0.f;
  if (i < n)
#pragma unroll 4
    for (int p = row; p < P; p += rows) s += src[p * ld + i];
  sh[threadIdx.x] = s;
  __syncthreads();
  for (int o = rows / 2; o > 0; o >>= 1) {
    if (row < o) sh[threadIdx.x] += sh[threadIdx.x + o * cols];
    __syncthreads();
  }
  if (row == 0 && i < n) grad[i] += sh[col];
}
constexpr int kBiasCols = 2;
__global__ void __launch_bounds__(256)
    k_sum_parts(const float* __restrict__ part, int P, long long n, int cols, float* __restrict__ grad,
                const float* __restrict__ part_b, int Pb, int nb, int ldb, float* __restrict__ grad_b) {
  const long long wb = (n + cols - 1) / cols;
  if (blockIdx.x < wb) sum_columns(part, P, n, n, cols, blockIdx.x, grad);
  else sum_columns(part_b, Pb, nb, ldb, kBiasCols, blockIdx.x - wb, grad_b);
}

// x (planes) to the channel-innermost BF16 input, padded channels 0; eight
// channels of a pixel per store
__global__ void __launch_bounds__(256) k_input(const float* __restrict__ x, int C, int CP, long long HW,
                                               bf16* __restrict__ o) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < HW;
       i += (long long)gridDim.x * blockDim.x)
    for (int c = 0; c < CP; c += 8) {
      bf162 v[4];
#pragma unroll
      for (int k = 0; k < 4; ++k)
        v[k] = __floats2bfloat162_rn(c + 2 * k < C ? x[(c + 2 * k) * HW + i] : 0.f,
                                     c + 2 * k + 1 < C ? x[(c + 2 * k + 1) * HW + i] : 0.f);
      *reinterpret_cast<uint4*>(o + i * CP + c) = *reinterpret_cast<const uint4*>(v);
    }
}

// dL/dy (planes) to the head's hi + lo pair, and its bias gradient partials
__global__ void __launch_bounds__(256) k_head_grad(const float* __restrict__ dy, int C, int CP,
                                                   long long HW, bf16* __restrict__ hi,
                                                   bf16* __restrict__ lo, float* __restrict__ part_b) {
  __shared__ float sh[8][8];
  for (int c = 0; c < CP; c += 8) {
    float s[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) s[k] = 0.f;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < HW;
         i += (long long)gridDim.x * blockDim.x) {
      bf162 h[4], l[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const float v0 = c + 2 * k < C ? dy[(c + 2 * k) * HW + i] : 0.f;
        const float v1 = c + 2 * k + 1 < C ? dy[(c + 2 * k + 1) * HW + i] : 0.f;
        split2(v0, v1, h[k], l[k]);
        s[2 * k] += v0;
        s[2 * k + 1] += v1;
      }
      *reinterpret_cast<uint4*>(hi + i * CP + c) = *reinterpret_cast<const uint4*>(h);
      *reinterpret_cast<uint4*>(lo + i * CP + c) = *reinterpret_cast<const uint4*>(l);
    }
#pragma unroll
    for (int k = 0; k < 8; ++k)
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) s[k] += __shfl_xor_sync(0xffffffffu, s[k], o);
    __syncthreads();
    if ((threadIdx.x & 31) == 0)
#pragma unroll
      for (int k = 0; k < 8; ++k) sh[threadIdx.x >> 5][k] = s[k];
    __syncthreads();
    if (threadIdx.x < 8) {
      float t = 0.f;
      for (int r = 0; r < 8; ++r) t += sh[r][threadIdx.x];
      part_b[(long long)blockIdx.x * CP + c + threadIdx.x] = t;
    }
  }
}

// The BF16 weights of every layer in the order the convolutions stage them:
// forward [16 co][chunk of 16 ci][tap][co][ci], data gradient
// [16 ci][chunk of 16 co][flipped tap][ci][co]; padded channels 0.
struct PackLayer {
  long long off_w, off_f, off_d;  // FP32 weights, packed forward, packed gradient
  int co, ca, cb, coP, caP, cbP, kk;
};
constexpr int kMaxLayers = 15;
struct PackTable {
  PackLayer l[kMaxLayers];
  int n;
};
__global__ void __launch_bounds__(256) k_pack(PackTable t, const float* __restrict__ w,
                                              bf16* __restrict__ wf, bf16* __restrict__ wd) {
  const PackLayer L = t.l[blockIdx.y];
  const int ciP = L.caP + L.cbP, ci = L.ca + L.cb;
  const long long n = (long long)L.coP * ciP * L.kk;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x) {
    const int k = int(i & 15), r = int((i >> 4) & 15);
    long long q = i >> 8;
    const int tap = int(q % L.kk);
    q /= L.kk;
    auto value = [&](int co, int cp, int tp) {
      const int c = cp < L.caP ? (cp < L.ca ? cp : -1) : (cp - L.caP < L.cb ? L.ca + cp - L.caP : -1);
      return co < L.co && c >= 0 ? w[L.off_w + ((long long)co * ci + c) * L.kk + tp] : 0.f;
    };
    const int kf = int(q % (ciP / 16)), gf = int(q / (ciP / 16));
    wf[L.off_f + i] = __float2bfloat16(value(gf * 16 + r, kf * 16 + k, tap));
    const int kd = int(q % (L.coP / 16)), gd = int(q / (L.coP / 16));
    wd[L.off_d + i] = __float2bfloat16(value(kd * 16 + k, gd * 16 + r, L.kk - 1 - tap));
  }
}

// Adam (Kingma & Ba) on the FP32 master weights.
__global__ void k_adam(float* __restrict__ w, float* __restrict__ m, float* __restrict__ v,
                       float* __restrict__ g, long long n, float lr, float b1, float b2, float eps,
                       float c1, float c2, float scale) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x) {
    const float gi = g[i] * scale;
    const float mi = b1 * m[i] + (1.f - b1) * gi;
    const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    w[i] = w[i] - lr * (mi / c1) / (sqrtf(vi / c2) + eps);
    g[i] = 0.f;
  }
}

// float(double(d) * inv) for inv = hi + lo + less than 2^-48 inv, in FP32: the
// product's leading part q and the rest r with an error below 2^-46 |q|.  Where
// that could change the rounding (one value in 2^20), and below 2^-100, where
// the parts leave FP32's range, the product is taken in FP64, in a call: as a
// selected value it would be computed for every d.
__device__ __noinline__ float scale_fp64(float d, double inv) { return float(double(d) * inv); }
__device__ __forceinline__ float scale_exact(float d, double inv, float hi, float lo) {
  const float q = __fmul_rn(d, hi);  // not fused with the additions below
  const float r = fmaf(d, lo, fmaf(d, hi, -q)), tol = fabsf(q) * 0x1p-45f;
  const float a = q + (r - tol), b = q + (r + tol);
  if ((fabsf(q) >= 0x1p-100f && a == b) || d == 0.f) return d == 0.f ? q : a;
  return scale_fp64(d, inv);
}

// masked MSE: loss partials per block, dy = (y - t) mask / n.  One FP64
// conversion and FMA per value (26 -> 12 us at 528 x 520, cold; with FP64 products and
// back-conversions that pipe was 81 % busy).
__global__ void __launch_bounds__(256) k_mse(const float* __restrict__ y, const float* __restrict__ t,
                                             const float* __restrict__ mask, int C, long long HW,
                                             double inv, float inv_hi, float inv_lo, float* __restrict__ dy,
                                             double* __restrict__ part) {
  double acc = 0.0;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < HW;
       i += (long long)gridDim.x * blockDim.x) {
    const float mk = mask ? mask[i] : 1.f;
    for (int c = 0; c < C; ++c) {
      const long long j = c * HW + i;
      const float d = (y[j] - t[j]) * mk;
      dy[j] = scale_exact(d, inv, inv_hi, inv_lo);
      acc += double(d) * double(d);
    }
  }
  __shared__ double sh[256];
  sh[threadIdx.x] = acc;
  __syncthreads();
  for (int s = 128; s > 0; s >>= 1) {
    if (threadIdx.x < s) sh[threadIdx.x] += sh[threadIdx.x + s];
    __syncthreads();
  }
  if (threadIdx.x == 0) part[blockIdx.x] = sh[0];
}

constexpr int kMaxGrid = 1216;  // eight 256-thread blocks per SM

int grid1(long long n) {
  long long b = (n + 255) / 256;
  if (b > kMaxGrid) b = kMaxGrid;
  return int(b < 1 ? 1 : b);
}

}  // namespace

// ------------------------------------------------------------------ network
struct ConvLayer {
  int co, ci, k;
  long long off_w, off_b;  // offsets into the parameter vector
  int ca, cb;              // input channels: first operand, concatenated skip
  int coP, caP, cbP;       // padded to 16
  long long off_f, off_d;  // packed weights, forward and data gradient
};

struct pf_unet {
  int H = 0, W = 0, nin = 0, nout = 0, L = 4;
  int sms = 1;  // SMs of the device (tile and chunk choices)
  int ch[4] = {16, 32, 64, 128};
  cudaStream_t st = nullptr;
  std::vector<ConvLayer> layers;  // enc0a, enc0b, ..., enc3b, dec2a, dec2b, dec1a, ..., head
  long long nparam = 0;
  float *w32 = nullptr, *m = nullptr, *v = nullptr, *g = nullptr;
  bf16 *wf = nullptr, *wd = nullptr;  // packed BF16 weights
  PackTable pack{};
  int adam_t = 0;
  bf16* xin = nullptr;                 // input, channel-innermost
  std::vector<bf16*> act;              // output of every 3x3 layer
  bf16* pool[3] = {nullptr, nullptr, nullptr};   // 2x2 average of encoder level k
  float* skip[3] = {nullptr, nullptr, nullptr};  // gradient of encoder level k through its skip
  std::vector<bf16*> dh, dl;           // dL/d(pre-activation) of every layer, hi and lo
  float* wpart = nullptr;              // weight-gradient partials
  std::vector<float*> bpart;           // bias-gradient partials of every layer
  // the backward pass's second stream: weight gradients beside the chain of
  // data gradients
  cudaStream_t side = nullptr;
  std::vector<cudaEvent_t> ev;         // layer l's gradient is written; last: the side stream is done
  double* lpart = nullptr;
  double* h_loss = nullptr;
  void* slab = nullptr;  // device memory of everything above
};

namespace {

int pad16(int c) { return (c + 15) / 16 * 16; }
long long conv_tiles(int H, int W) { return (long long)((W + TW - 1) / TW) * ((H + TH - 1) / TH); }

// resolution of layer l's output: level of the layer
int layer_level(const pf_unet* u, int l) {
  if (l < 2 * u->L) return l / 2;
  const int d = l - 2 * u->L;  // decoder index 0 .. 2(L-1)-1 (+ head)
  if (d >= 2 * (u->L - 1)) return 0;
  return u->L - 2 - d / 2;
}
bool is_head(const pf_unet* u, int l) { return l == int(u->layers.size()) - 1; }
bool reads_pool(const pf_unet* u, int l) { return l > 0 && l < 2 * u->L && l % 2 == 0; }
// first convolution of a decoder level: [up(below), skip of level k]
bool reads_up(const pf_unet* u, int l) { return l >= 2 * u->L && !is_head(u, l) && (l - 2 * u->L) % 2 == 0; }

ConvSrc layer_input(const pf_unet* u, int l) {
  ConvSrc in{};
  const ConvLayer& c = u->layers[l];
  in.ca = c.caP;
  in.cb = c.cbP;
  if (l == 0) {
    in.a = u->xin;
  } else if (reads_pool(u, l)) {
    in.a = u->pool[l / 2 - 1];
  } else {
    in.a = u->act[l - 1];
    if (reads_up(u, l)) {
      in.up = 1;
      in.b = u->act[2 * layer_level(u, l) + 1];
    }
  }
  return in;
}

cudaError_t pack_weights(pf_unet* u) {
  k_pack<<<dim3(256, u->pack.n), 256, 0, u->st>>>(u->pack, u->w32, u->wf, u->wd);
  return cudaGetLastError();
}

}  // namespace

extern "C" {

pf_status pf_unet_destroy(pf_unet* u) {
  if (!u) return PF_OK;
  if (u->st) cudaStreamSynchronize(u->st);
  else cudaDeviceSynchronize();
  if (u->side) {
    cudaStreamSynchronize(u->side);
    cudaStreamDestroy(u->side);
  }
  for (cudaEvent_t e : u->ev) cudaEventDestroy(e);
  if (u->slab) cudaFree(u->slab);
  if (u->h_loss) cudaFreeHost(u->h_loss);
  delete u;
  return PF_OK;
}

pf_status pf_unet_create(int height, int width, int n_in, int n_out, const int channels[4],
                         void* stream, pf_unet** out) {
  if (!out || !channels) {
    set_error("unet_create: null argument");
    return PF_EINVAL;
  }
  *out = nullptr;
  if (height < 8 || width < 8 || height % 8 || width % 8 || height > 16384 || width > 16384 ||
      n_in < 1 || n_in > 64 || n_out < 1 || n_out > 64) {
    set_error("unet_create: height and width must be multiples of 8 (8 .. 16384); 1 .. 64 channels in/out");
    return PF_EINVAL;
  }
  for (int k = 0; k < 4; ++k)
    if (channels[k] < 1 || channels[k] > 512) {
      set_error("unet_create: channels must be 1 .. 512");
      return PF_EINVAL;
    }
  pf_unet* u = new pf_unet();
  u->H = height; u->W = width; u->nin = n_in; u->nout = n_out;
  {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&u->sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
      u->sms = 1;
  }
  for (int k = 0; k < 4; ++k) u->ch[k] = channels[k];
  u->st = static_cast<cudaStream_t>(stream);
  long long off = 0, off_p = 0;
  auto add = [&](int co, int ca, int cb, int k) {
    ConvLayer c{};
    c.co = co; c.ci = ca + cb; c.k = k; c.ca = ca; c.cb = cb;
    c.coP = pad16(co); c.caP = pad16(ca); c.cbP = pad16(cb);
    c.off_w = off;
    c.off_b = off + (long long)co * c.ci * k * k;
    off = c.off_b + co;
    c.off_f = c.off_d = off_p;
    off_p += (long long)c.coP * (c.caP + c.cbP) * k * k;
    u->layers.push_back(c);
  };
  int cprev = n_in;
  for (int k = 0; k < 4; ++k) {
    add(u->ch[k], cprev, 0, 3);
    add(u->ch[k], u->ch[k], 0, 3);
    cprev = u->ch[k];
  }
  for (int k = 2; k >= 0; --k) {
    add(u->ch[k], u->ch[k + 1], u->ch[k], 3);
    add(u->ch[k], u->ch[k], 0, 3);
  }
  add(n_out, u->ch[0], 0, 1);
  u->nparam = off;
  for (const ConvLayer& c : u->layers)
    u->pack.l[u->pack.n++] = PackLayer{c.off_w, c.off_f, c.off_d, c.co, c.ca, c.cb, c.coP, c.caP, c.cbP, c.k * c.k};
  const long long HW = (long long)height * width;
  std::vector<std::pair<void**, size_t>> need;
  auto want = [&](void* p, size_t bytes) { need.push_back({static_cast<void**>(p), bytes}); };
  want(&u->w32, sizeof(float) * off);
  want(&u->m, sizeof(float) * off);
  want(&u->v, sizeof(float) * off);
  want(&u->g, sizeof(float) * off);
  want(&u->wf, sizeof(bf16) * off_p);
  want(&u->wd, sizeof(bf16) * off_p);
  want(&u->xin, sizeof(bf16) * pad16(n_in) * HW);
  want(&u->lpart, sizeof(double) * kMaxGrid);
  const int nl = int(u->layers.size());
  u->act.assign(nl - 1, nullptr);
  u->dh.assign(nl, nullptr);
  u->dl.assign(nl, nullptr);
  u->bpart.assign(nl, nullptr);
  long long max_part = 0;
  for (int l = 0; l < nl; ++l) {
    const int lev = layer_level(u, l);
    const int Hl = height >> lev, Wl = width >> lev;
    const long long hw = HW >> (2 * lev);
    const ConvLayer& c = u->layers[l];
    if (l < nl - 1) want(&u->act[l], sizeof(bf16) * c.coP * hw);
    want(&u->dh[l], sizeof(bf16) * c.coP * hw);
    want(&u->dl[l], sizeof(bf16) * c.coP * hw);
    const int P = wgrad_chunks(Hl, Wl, c.caP + c.cbP, c.coP, u->sms);
    max_part = std::max(max_part, (long long)P * c.co * c.ci * c.k * c.k);
    // bias partials: one row per tile of the data gradient of the layer above
    const int la = l < nl - 1 ? layer_level(u, l + 1) : 0;
    const long long rows = l < nl - 1 ? conv_tiles(height >> la, width >> la) : kMaxGrid;
    want(&u->bpart[l], sizeof(float) * rows * c.coP);
  }
  for (int k = 0; k < 3; ++k) {
    want(&u->pool[k], sizeof(bf16) * pad16(u->ch[k]) * (HW >> (2 * k + 2)));
    want(&u->skip[k], sizeof(float) * pad16(u->ch[k]) * (HW >> (2 * k)));
  }
  want(&u->wpart, sizeof(float) * max_part);
  // one allocation for all of them, each on a 256-byte boundary
  size_t total = 0;
  for (auto& n : need) total += (n.second + 255) / 256 * 256;
  if (cudaMalloc((void**)&u->slab, total) != cudaSuccess) {
    pf_unet_destroy(u);
    set_error("unet: cudaMalloc failed");
    return PF_ENOMEM;
  }
  cudaMemsetAsync(u->slab, 0, total, u->st);
  total = 0;
  for (auto& n : need) {
    *n.first = static_cast<char*>(u->slab) + total;
    total += (n.second + 255) / 256 * 256;
  }
  bool ok = cudaStreamCreateWithFlags(&u->side, cudaStreamNonBlocking) == cudaSuccess;
  for (int l = 0; l <= nl && ok; ++l) {
    cudaEvent_t e = nullptr;
    ok = cudaEventCreateWithFlags(&e, cudaEventDisableTiming) == cudaSuccess;
    if (ok) u->ev.push_back(e);
  }
  if (!ok) {
    pf_unet_destroy(u);
    set_error("unet_create: stream or event creation failed");
    return PF_ECUDA;
  }
  if (cudaMallocHost((void**)&u->h_loss, sizeof(double) * kMaxGrid) != cudaSuccess) {
    pf_unet_destroy(u);
    set_error("unet_create: cudaMallocHost failed");
    return PF_ENOMEM;
  }
  if (cudaStreamSynchronize(u->st) != cudaSuccess) {
    pf_unet_destroy(u);
    set_error("unet_create: stream error");
    return PF_ECUDA;
  }
  *out = u;
  return PF_OK;
}

pf_status pf_unet_num_params(const pf_unet* u, long long* n) {
  if (!u || !n) {
    set_error("unet_num_params: null argument");
    return PF_EINVAL;
  }
  *n = u->nparam;
  return PF_OK;
}

pf_status pf_unet_set_params(pf_unet* u, const float* params) {
  if (!u || !params) {
    set_error("unet_set_params: null argument");
    return PF_EINVAL;
  }
  cudaError_t e = cudaMemcpyAsync(u->w32, params, sizeof(float) * u->nparam, cudaMemcpyHostToDevice, u->st);
  if (e == cudaSuccess) {
    e = pack_weights(u);
    cudaMemsetAsync(u->m, 0, sizeof(float) * u->nparam, u->st);
    cudaMemsetAsync(u->v, 0, sizeof(float) * u->nparam, u->st);
    cudaMemsetAsync(u->g, 0, sizeof(float) * u->nparam, u->st);
    u->adam_t = 0;
    if (e == cudaSuccess) e = cudaStreamSynchronize(u->st);
  }
  if (e != cudaSuccess) {
    set_error(std::string("unet_set_params: ") + cudaGetErrorString(e));
    return PF_ECUDA;
  }
  return PF_OK;
}

static pf_status copy_out(pf_unet* u, const float* src, float* dst, const char* what) {
  if (!u || !dst) {
    set_error(std::string(what) + ": null argument");
    return PF_EINVAL;
  }
  cudaError_t e = cudaMemcpyAsync(dst, src, sizeof(float) * u->nparam, cudaMemcpyDeviceToHost, u->st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(u->st);
  if (e != cudaSuccess) {
    set_error(std::string(what) + ": " + cudaGetErrorString(e));
    return PF_ECUDA;
  }
  return PF_OK;
}

pf_status pf_unet_get_params(pf_unet* u, float* params) { return copy_out(u, u ? u->w32 : nullptr, params, "unet_get_params"); }
pf_status pf_unet_get_grads(pf_unet* u, float* grads) { return copy_out(u, u ? u->g : nullptr, grads, "unet_get_grads"); }

pf_status pf_unet_forward(pf_unet* u, const float* x, float* y) {
  if (!u || !x || !y) {
    set_error("unet_forward: null argument");
    return PF_EINVAL;
  }
  const long long HW = (long long)u->H * u->W;
  k_input<<<grid1(HW), 256, 0, u->st>>>(x, u->nin, pad16(u->nin), HW, u->xin);
  cudaError_t e = cudaGetLastError();
  const int nl = int(u->layers.size());
  for (int l = 0; l < nl && e == cudaSuccess; ++l) {
    const ConvLayer& c = u->layers[l];
    const int lev = layer_level(u, l);
    const int H = u->H >> lev, W = u->W >> lev, KC = (c.caP + c.cbP) / 16;
    const ConvSrc in = layer_input(u, l);
    EpiArgs a{};
    a.bias = u->w32 + c.off_b;
    a.co = c.co;
    a.cp = c.coP;
    if (is_head(u, l)) {
      a.y = y;
      e = launch_conv<1, EPI_HEAD>(in, nullptr, u->wf + c.off_f, H, W, c.coP, KC, a, u->sms, u->st);
    } else {
      a.out = u->act[l];
      if (l < 2 * u->L && l % 2 == 1 && lev < u->L - 1) a.pool = u->pool[lev];
      e = launch_conv<3, EPI_FWD>(in, nullptr, u->wf + c.off_f, H, W, c.coP, KC, a, u->sms, u->st);
    }
  }
  if (e != cudaSuccess) {
    set_error(std::string("unet_forward: ") + cudaGetErrorString(e));
    return PF_ECUDA;
  }
  return PF_OK;
}

// Backward from dL/dy (FP32, n_out x H x W); parameter gradients are added to
// the accumulated gradient (zeroed by pf_unet_adam or pf_unet_set_params).
pf_status pf_unet_backward(pf_unet* u, const float* dy) {
  if (!u || !dy) {
    set_error("unet_backward: null argument");
    return PF_EINVAL;
  }
  const int nl = int(u->layers.size());
  const long long HW = (long long)u->H * u->W;
  int Pb = grid1(HW);  // bias partials of layer l
  k_head_grad<<<Pb, 256, 0, u->st>>>(dy, u->nout, u->layers[nl - 1].coP, HW, u->dh[nl - 1], u->dl[nl - 1],
                                     u->bpart[nl - 1]);
  cudaError_t e = cudaGetLastError();
  for (int l = nl - 1; l >= 0 && e == cudaSuccess; --l) {
    const ConvLayer& c = u->layers[l];
    const int lev = layer_level(u, l);
    const int H = u->H >> lev, W = u->W >> lev;
    const ConvSrc in = layer_input(u, l);
    const bf16 *dh = u->dh[l], *dl = u->dl[l];
    // weight and bias gradients, on the side stream once this layer's
    // gradient is written (the deep levels' launches leave most SMs idle)
    if ((e = cudaEventRecord(u->ev[l], u->st)) != cudaSuccess) break;
    if ((e = cudaStreamWaitEvent(u->side, u->ev[l], 0)) != cudaSuccess) break;
    const int P = wgrad_chunks(H, W, c.caP + c.cbP, c.coP, u->sms);
    const long long nw = (long long)c.co * c.ci * c.k * c.k;
    e = c.k == 3 ? launch_wgrad<3>(dh, dl, c.coP, in, c.ca, c.cb, H, W, c.co, P, u->wpart, u->side)
                 : launch_wgrad<1>(dh, dl, c.coP, in, c.ca, c.cb, H, W, c.co, P, u->wpart, u->side);
    if (e != cudaSuccess) break;
    // narrow blocks where there are many partials: backward at 136^2 274 us
    // against 280 with 32 columns throughout (and 338 with 8), 394 against 393 at
    // 264^2, 714 against 698 at 528 x 520
    const int cols = P >= 64 ? 8 : 32;
    k_sum_parts<<<unsigned((nw + cols - 1) / cols + (c.co + kBiasCols - 1) / kBiasCols), 256, 0, u->side>>>(
        u->wpart, P, nw, cols, u->g + c.off_w, u->bpart[l], Pb, c.co, c.coP, u->g + c.off_b);
    e = cudaGetLastError();
    if (l == 0 || e != cudaSuccess) continue;  // no gradient needed for the input features
    // data gradient, down to dL/d(pre-activation) of layer l - 1
    const ConvLayer& b = u->layers[l - 1];
    ConvSrc s{};
    s.a = dh;
    s.ca = c.coP;
    EpiArgs a{};
    a.cp = b.coP;
    a.act = u->act[l - 1];
    a.hi = u->dh[l - 1];
    a.lo = u->dl[l - 1];
    a.part_b = u->bpart[l - 1];
    const bf16* w = u->wd + c.off_d;
    const int KC = c.coP / 16, N = c.caP + c.cbP;
    if (reads_up(u, l)) {
      a.ca = c.caP;
      a.cb = c.cbP;
      a.skip_out = u->skip[lev];
      e = launch_conv<3, EPI_UP>(s, dl, w, H, W, N, KC, a, u->sms, u->st);
    } else if (reads_pool(u, l)) {
      a.skip_in = u->skip[lev - 1];
      e = launch_conv<3, EPI_POOL>(s, dl, w, H, W, N, KC, a, u->sms, u->st);
    } else if (is_head(u, l)) {
      e = launch_conv<1, EPI_PLAIN>(s, dl, w, H, W, N, KC, a, u->sms, u->st);
    } else {
      e = launch_conv<3, EPI_PLAIN>(s, dl, w, H, W, N, KC, a, u->sms, u->st);
    }
    Pb = int(conv_tiles(H, W));
  }
  // the caller's stream goes on once every gradient is added (also after a
  // failed launch: what was started must not outlive the call's order)
  const cudaError_t ej = cudaEventRecord(u->ev[nl], u->side);
  const cudaError_t ew = cudaStreamWaitEvent(u->st, u->ev[nl], 0);
  if (e == cudaSuccess) e = ej != cudaSuccess ? ej : ew;
  if (e != cudaSuccess) {
    set_error(std::string("unet_backward: ") + cudaGetErrorString(e));
    return PF_ECUDA;
  }
  return PF_OK;
}

pf_status pf_unet_adam(pf_unet* u, float lr, float beta1, float beta2, float eps, float grad_scale) {
  if (!u || !(lr > 0) || !(beta1 >= 0 && beta1 < 1) || !(beta2 >= 0 && beta2 < 1) || !(eps > 0)) {
    set_error("unet_adam: bad argument");
    return PF_EINVAL;
  }
  u->adam_t += 1;
  const float c1 = 1.f - std::pow(beta1, float(u->adam_t)), c2 = 1.f - std::pow(beta2, float(u->adam_t));
  k_adam<<<grid1(u->nparam), 256, 0, u->st>>>(u->w32, u->m, u->v, u->g, u->nparam, lr, beta1, beta2,
                                               eps, c1, c2, grad_scale);
  cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess) e = pack_weights(u);
  if (e != cudaSuccess) {
    set_error(std::string("unet_adam: ") + cudaGetErrorString(e));
    return PF_ECUDA;
  }
  return PF_OK;
}

pf_status pf_unet_mse(pf_unet* u, const float* y, const float* t, const float* mask,
                      double n_valid, float* dy, double* loss) {
  if (!u || !y || !t || !dy || !loss || !(n_valid > 0)) {
    set_error("unet_mse: bad argument");
    return PF_EINVAL;
  }
  const long long HW = (long long)u->H * u->W;
  const double n = double(u->nout) * (mask ? n_valid : double(HW));
  const int nb = grid1(HW);
  const double inv = 1.0 / n;
  k_mse<<<nb, 256, 0, u->st>>>(y, t, mask, u->nout, HW, inv, float(inv), float(inv - double(float(inv))), dy,
                               u->lpart);
  cudaError_t e = cudaMemcpyAsync(u->h_loss, u->lpart, sizeof(double) * nb, cudaMemcpyDeviceToHost, u->st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(u->st);
  if (e != cudaSuccess) {
    set_error(std::string("unet_mse: ") + cudaGetErrorString(e));
    return PF_ECUDA;
  }
  double s = 0;
  for (int i = 0; i < nb; ++i) s += u->h_loss[i];
  *loss = 0.5 * s * inv;
  return PF_OK;
}

}  // extern "C"
