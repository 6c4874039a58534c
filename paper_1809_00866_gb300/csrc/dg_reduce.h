// Fixed-order FP64 sums of up to eight dot products at a time over the threads of a CTA.
#pragma once

#include <cuda_runtime.h>

namespace dg {

// Sums acc[0..8) over the warp's lanes by halving: every step swaps the half of the values that the
// other lane keeps, so eight sums take 9 additions instead of the 40 of eight butterflies (an FP64
// addition holds GB300's FP64 pipe as long as a multiply-add: the butterflies were 38 % of the
// pipe's work in the dot products; with them and 608 chunks instead of 2240, eight dot products at 32^3 P4
// 172 -> 71 us, their partial sums 29 -> 10 us). Lane l holds the sum of value (l >> 2).
__device__ __forceinline__ double warp_sum8(double (&acc)[8], int lane) {
  double a4[4], a2[2], a1;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const double keep = lane & 16 ? acc[k + 4] : acc[k], send = lane & 16 ? acc[k] : acc[k + 4];
    a4[k] = keep + __shfl_xor_sync(0xffffffffu, send, 16);
  }
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    const double keep = lane & 8 ? a4[k + 2] : a4[k], send = lane & 8 ? a4[k] : a4[k + 2];
    a2[k] = keep + __shfl_xor_sync(0xffffffffu, send, 8);
  }
  {
    const double keep = lane & 4 ? a2[1] : a2[0], send = lane & 4 ? a2[0] : a2[1];
    a1 = keep + __shfl_xor_sync(0xffffffffu, send, 4);
  }
  a1 += __shfl_xor_sync(0xffffffffu, a1, 2);
  a1 += __shfl_xor_sync(0xffffffffu, a1, 1);
  return a1;
}

// Sum of one value over the warp (every lane gets it).
__device__ __forceinline__ double warp_sum(double a) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
  return a;
}

// Dot products of w[i0, i1) with nv <= 8 vectors V, V + ldv, ... by a CTA of NT threads: thread v < nv
// returns the sum for vector v (red: [NT / 32][8] shared doubles; two barriers).
template <int NT>
__device__ __forceinline__ double block_dots(const double* __restrict__ V, long long ldv, int nv,
                                             const double* __restrict__ w, long long i0, long long i1, long long step,
                                             double (&red)[NT / 32][8]) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  double out = 0.0;
  if (nv == 1) {
    double a = 0.0;
    for (long long i = i0 + threadIdx.x; i < i1; i += step) a += V[i] * w[i];
    a = warp_sum(a);
    if (lane == 0) red[warp][0] = a;
  } else {
    double acc[8];
#pragma unroll
    for (int v = 0; v < 8; ++v) acc[v] = 0.0;
    long long i = i0 + threadIdx.x;
    for (; i + step < i1; i += 2 * step) {  // two entries of every vector in flight
      const double w0 = w[i], w1 = w[i + step];
      double a[8], b[8];
#pragma unroll
      for (int v = 0; v < 8; ++v)
        if (v < nv) {
          a[v] = V[(size_t)v * ldv + i];
          b[v] = V[(size_t)v * ldv + i + step];
        }
#pragma unroll
      for (int v = 0; v < 8; ++v)
        if (v < nv) acc[v] += a[v] * w0;
#pragma unroll
      for (int v = 0; v < 8; ++v)
        if (v < nv) acc[v] += b[v] * w1;
    }
    if (i < i1) {
      const double w0 = w[i];
#pragma unroll
      for (int v = 0; v < 8; ++v)
        if (v < nv) acc[v] += V[(size_t)v * ldv + i] * w0;
    }
    const double s = warp_sum8(acc, lane);
    if ((lane & 3) == 0) red[warp][lane >> 2] = s;
  }
  __syncthreads();
  if (threadIdx.x < nv) {
#pragma unroll
    for (int q = 0; q < NT / 32; ++q) out += red[q][threadIdx.x];
  }
  __syncthreads();
  return out;
}

}  // namespace dg
