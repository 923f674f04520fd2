// y = S v for a 3^d-point block stencil S[((o F + f) F + h) N + i] on grids
// where one thread per output row leaves the chip waiting on latency: a row
// is shared by 3 (2D) or 9 (3D) threads, one per line of three offsets along
// x, whose partial sums are added in shared memory in ascending order.  A
// thread then has 9 or 12 independent pairs of loads and as many FMAs in
// F short chains (an FP64 FMA's result is ready after several times its issue
// slot); a neighbour outside the grid is read at the node itself and counted
// as 0, so no load waits for a branch.  One thread per row walking its 27 or
// 108 entries took 9.5 us for the 9,315 FP64 rows of 69 x 45 nodes and 74 us
// for the 143,748 FP32 rows of 33^3 (ncu, cold cache); now 6.5 and 17.6 us.
// A launch starts while the one before it drains (launch_dependent).
#pragma once
#include <cuda_runtime.h>

#include "pf_internal.h"
#include "pf_launch.cuh"

namespace pf {

template <int D>
struct StencilRows {
  static constexpr int LINES = D == 3 ? 9 : 3, LANES = D == 3 ? 32 : 64;
  static constexpr int THREADS = LINES * LANES;
};

template <int D, class TS, class TV>
__global__ void __launch_bounds__(StencilRows<D>::THREADS)
    k_stencil_rows(Geom g, const TS* S, const TV* v, TV* y, const int* skip) {
  launch_wait();
  if (skip && *skip) return;
  constexpr int F = D + 1, LINES = StencilRows<D>::LINES, LANES = StencilRows<D>::LANES;
  __shared__ TV part[LINES][LANES];
  const int lane = threadIdx.x % LANES, line = threadIdx.x / LANES;
  const int dy = line % 3 - 1, dz = D == 3 ? line / 3 - 1 : 0;
  const long long N = g.N, total = F * N;
  const long long t = blockIdx.x * (long long)LANES + lane;
  TV sum = TV(0);
  if (t < total) {
    const int f = int(t / N);
    const long long i = t - (long long)f * N;
    const long long plane = (long long)g.n[0] * g.n[1];
    int ix, iy, iz = 0;
    if (N <= 0xffffffffLL) {
      const unsigned r = D == 3 ? unsigned(i) % unsigned(plane) : unsigned(i);
      if (D == 3) iz = int(unsigned(i) / unsigned(plane));
      iy = int(r / unsigned(g.n[0]));
      ix = int(r % unsigned(g.n[0]));
    } else {
      const long long r = D == 3 ? i % plane : i;
      if (D == 3) iz = int(i / plane);
      iy = int(r / g.n[0]);
      ix = int(r % g.n[0]);
    }
    const bool in_line = iy + dy >= 0 && iy + dy < g.n[1] && iz + dz >= 0 && iz + dz < g.n[2];
    const TV* p = v + i + (in_line ? dy * (long long)g.n[0] + dz * plane : 0);
    const bool in[3] = {in_line && ix > 0, in_line, in_line && ix + 1 < g.n[0]};
    const TS* s = S + ((long long)line * 3 * F + f) * F * N + i;
    TS a[3][F];
    TV w[3][F];
#pragma unroll
    for (int k = 0; k < 3; ++k)
#pragma unroll
      for (int h = 0; h < F; ++h) {
        a[k][h] = s[(long long)(k * F * F + h) * N];
        w[k][h] = p[(in[k] ? k - 1 : 0) + h * N];
      }
    TV acc[F];
#pragma unroll
    for (int h = 0; h < F; ++h) acc[h] = TV(a[0][h]) * (in[0] ? w[0][h] : TV(0));
#pragma unroll
    for (int k = 1; k < 3; ++k)
#pragma unroll
      for (int h = 0; h < F; ++h) acc[h] += TV(a[k][h]) * (in[k] ? w[k][h] : TV(0));
    sum = F == 4 ? (acc[0] + acc[1]) + (acc[2] + acc[F - 1]) : (acc[0] + acc[1]) + acc[2];
  }
  part[line][lane] = sum;
  __syncthreads();
  if (line == 0 && t < total) {
#pragma unroll
    for (int l = 1; l < LINES; ++l) sum += part[l][lane];
    y[t] = sum;
  }
}

// Launch over all rows; cudaErrorInvalidConfiguration beyond 2^31 blocks.
template <int D, class TS, class TV>
inline cudaError_t stencil_rows(const Geom& g, const TS* S, const TV* v, TV* y, cudaStream_t st,
                                const int* skip) {
  using R = StencilRows<D>;
  const long long nb = ((D + 1) * g.N + R::LANES - 1) / R::LANES;
  if (nb > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
  return launch_dependent(k_stencil_rows<D, TS, TV>, dim3(unsigned(nb)), dim3(R::THREADS), st, g, S, v, y, skip);
}

}  // namespace pf
