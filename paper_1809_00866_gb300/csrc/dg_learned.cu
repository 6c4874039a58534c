// Learned coarse-level correction (no counterpart in the paper): a per-element network
// 112 -> 128 -> 128 -> 16 with GELU that maps the coarsest-level (P1) right-hand side of an
// element and of its six face neighbours to the element's correction. Inference and training
// run on the tensor cores with BF16 operands and FP32 accumulation (mma.sync m16n8k16); the
// packed BF16 weights reach shared memory by one bulk asynchronous copy (cp.async.bulk) that
// overlaps the gather of the features.
#include <cuda_bf16.h>

#include <cmath>
#include <cstdint>
#include <cstring>
#include <mutex>
#include <vector>

#include "dg_async.h"
#include "dg_internal.h"
#include "dg_launch.h"

namespace dg {

namespace {

constexpr int kIn = DG_MLP_IN, kHid = DG_MLP_HIDDEN, kOut = DG_MLP_OUT;
// offsets of the FP32 parameter vector theta
constexpr int oW1 = 0, ob1 = oW1 + kHid * kIn, oW2 = ob1 + kHid, ob2 = oW2 + kHid * kHid, oW3 = ob2 + kHid,
              ob3 = oW3 + kOut * kHid, kNP = ob3 + kOut;
static_assert(kNP == DG_MLP_NPARAM, "parameter count");

// Packed BF16 network (device and shared memory): rows padded to 120 / 136 entries so that
// the fragment loads of a warp hit 32 different banks; biases b1, b2, b3 in FP32 at the end.
constexpr int kLd1 = 120, kLd2 = 136;
constexpr int kPW1 = 0;
constexpr int kPW2 = kPW1 + kHid * kLd1 * 2;
constexpr int kPW3 = kPW2 + kHid * kLd2 * 2;
constexpr int kPB = kPW3 + kOut * kLd2 * 2;
constexpr int kPBytes = kPB + (2 * kHid + kOut) * 4;
static_assert(kPW2 % 16 == 0 && kPW3 % 16 == 0 && kPB % 16 == 0 && kPBytes % 16 == 0, "16-byte parts");

constexpr int kWarps = 4, kRows = 16 * kWarps;  // rows (elements or samples) per CTA

// ---------------------------------------------------------------- PTX helpers
// D += A B, m16n8k16, A row-major bf16, B column-major bf16, FP32 accumulators
__device__ __forceinline__ void mma16816(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%0,%1,%2,%3};\n"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// two floats -> packed bf16x2 (round to nearest even), the first in the low half
__device__ __forceinline__ uint32_t pack2(float lo, float hi) {
  __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  uint32_t u;
  memcpy(&u, &v, 4);
  return u;
}
__device__ __forceinline__ uint16_t bf16_bits(float x) {
  __nv_bfloat16 v = __float2bfloat16_rn(x);
  uint16_t u;
  memcpy(&u, &v, 2);
  return u;
}
__device__ __forceinline__ float bf16_to_f(uint16_t u) {
  return __uint_as_float(static_cast<uint32_t>(u) << 16);
}

constexpr float kRsqrt2 = 0.70710678118654752f, kRsqrt2Pi = 0.39894228040143268f;
__device__ __forceinline__ float gelu(float z) { return 0.5f * z * (1.0f + erff(z * kRsqrt2)); }
__device__ __forceinline__ float gelu_d(float z) {
  return 0.5f * (1.0f + erff(z * kRsqrt2)) + z * kRsqrt2Pi * expf(-0.5f * z * z);
}

// theta (FP32) -> packed BF16 network; one thread per packed slot
__global__ void pack_kernel(const float* __restrict__ theta, unsigned char* __restrict__ net) {
  if (!wait_previous()) return;
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  uint16_t* W1 = reinterpret_cast<uint16_t*>(net + kPW1);
  uint16_t* W2 = reinterpret_cast<uint16_t*>(net + kPW2);
  uint16_t* W3 = reinterpret_cast<uint16_t*>(net + kPW3);
  float* B = reinterpret_cast<float*>(net + kPB);
  if (i < kHid * kLd1) {
    const int r = i / kLd1, c = i % kLd1;
    W1[i] = c < kIn ? bf16_bits(theta[oW1 + r * kIn + c]) : 0;
    return;
  }
  i -= kHid * kLd1;
  if (i < kHid * kLd2) {
    const int r = i / kLd2, c = i % kLd2;
    W2[i] = c < kHid ? bf16_bits(theta[oW2 + r * kHid + c]) : 0;
    return;
  }
  i -= kHid * kLd2;
  if (i < kOut * kLd2) {
    const int r = i / kLd2, c = i % kLd2;
    W3[i] = c < kHid ? bf16_bits(theta[oW3 + r * kHid + c]) : 0;
    return;
  }
  i -= kOut * kLd2;
  if (i < kHid) B[i] = theta[ob1 + i];
  else if (i < 2 * kHid) B[i] = theta[ob2 + i - kHid];
  else if (i < 2 * kHid + kOut) B[i] = theta[ob3 + i - 2 * kHid];
}
constexpr int kPackSlots = kHid * kLd1 + kHid * kLd2 + kOut * kLd2 + 2 * kHid + kOut;

// Layers 2 and 3 and the bias/GELU epilogues of one warp's 16 rows, from the layer-1
// accumulators; out[j][.] holds the output columns 8j + 2t, 8j + 2t + 1 of rows g, g + 8.
__device__ __forceinline__ void mlp_tail(const unsigned char* sm, int g, int t, float (&acc)[16][4],
                                         float (&out)[2][4]) {
  const uint16_t* W2s = reinterpret_cast<const uint16_t*>(sm + kPW2);
  const uint16_t* W3s = reinterpret_cast<const uint16_t*>(sm + kPW3);
  const float* Bs = reinterpret_cast<const float*>(sm + kPB);
  uint32_t a[8][4];
#pragma unroll
  for (int kk = 0; kk < 8; ++kk) {
    a[kk][0] = pack2(gelu(acc[2 * kk][0]), gelu(acc[2 * kk][1]));
    a[kk][1] = pack2(gelu(acc[2 * kk][2]), gelu(acc[2 * kk][3]));
    a[kk][2] = pack2(gelu(acc[2 * kk + 1][0]), gelu(acc[2 * kk + 1][1]));
    a[kk][3] = pack2(gelu(acc[2 * kk + 1][2]), gelu(acc[2 * kk + 1][3]));
  }
#pragma unroll
  for (int j = 0; j < 16; ++j) {
    const float2 bb = *reinterpret_cast<const float2*>(Bs + kHid + 8 * j + 2 * t);
    acc[j][0] = bb.x; acc[j][1] = bb.y; acc[j][2] = bb.x; acc[j][3] = bb.y;
  }
#pragma unroll
  for (int kk = 0; kk < 8; ++kk)
#pragma unroll
    for (int j = 0; j < 16; ++j) {
      const uint32_t* w = reinterpret_cast<const uint32_t*>(W2s + (8 * j + g) * kLd2 + 16 * kk + 2 * t);
      mma16816(acc[j], a[kk], w[0], w[4]);
    }
#pragma unroll
  for (int kk = 0; kk < 8; ++kk) {
    a[kk][0] = pack2(gelu(acc[2 * kk][0]), gelu(acc[2 * kk][1]));
    a[kk][1] = pack2(gelu(acc[2 * kk][2]), gelu(acc[2 * kk][3]));
    a[kk][2] = pack2(gelu(acc[2 * kk + 1][0]), gelu(acc[2 * kk + 1][1]));
    a[kk][3] = pack2(gelu(acc[2 * kk + 1][2]), gelu(acc[2 * kk + 1][3]));
  }
#pragma unroll
  for (int j = 0; j < 2; ++j) {
    const float2 bb = *reinterpret_cast<const float2*>(Bs + 2 * kHid + 8 * j + 2 * t);
    out[j][0] = bb.x; out[j][1] = bb.y; out[j][2] = bb.x; out[j][3] = bb.y;
  }
#pragma unroll
  for (int kk = 0; kk < 8; ++kk)
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const uint32_t* w = reinterpret_cast<const uint32_t*>(W3s + (8 * j + g) * kLd2 + 16 * kk + 2 * t);
      mma16816(out[j], a[kk], w[0], w[4]);
    }
}

__device__ __forceinline__ void layer1(const unsigned char* sm, int g, int t, const uint32_t (&a1)[7][4],
                                       float (&acc)[16][4]) {
  const uint16_t* W1s = reinterpret_cast<const uint16_t*>(sm + kPW1);
  const float* Bs = reinterpret_cast<const float*>(sm + kPB);
#pragma unroll
  for (int j = 0; j < 16; ++j) {
    const float2 bb = *reinterpret_cast<const float2*>(Bs + 8 * j + 2 * t);
    acc[j][0] = bb.x; acc[j][1] = bb.y; acc[j][2] = bb.x; acc[j][3] = bb.y;
  }
#pragma unroll
  for (int kk = 0; kk < 7; ++kk)
#pragma unroll
    for (int j = 0; j < 16; ++j) {
      const uint32_t* w = reinterpret_cast<const uint32_t*>(W1s + (8 * j + g) * kLd1 + 16 * kk + 2 * t);
      mma16816(acc[j], a1[kk], w[0], w[4]);
    }
}

// Start the bulk copy of the packed network into shared memory (thread 0) and return.
__device__ __forceinline__ void start_weights(unsigned char* sm, const unsigned char* net, uint64_t* bar) {
  if (threadIdx.x == 0) mbar_init(bar, 1);
  __syncthreads();
  if (threadIdx.x == 0) {
    mbar_expect_tx(bar, kPBytes);
    bulk_g2s(sm, net, kPBytes, bar);
  }
}

// ------------------------------------------------------------- inference
// Rows of 16 features-times-7 (FEAT: given features X [n][112] -> Y [n][16]) or the coarse
// correction (COARSE: gathered from the level vector d [ne][16] and neighbours nbr [ne][6],
// normalised, x = s N(X)). One warp per 16 rows, 4 warps per CTA.
enum { kModeFeat = 0, kModeCoarse = 1 };

template <int MODE, class R>
__global__ void __launch_bounds__(32 * kWarps) mlp_forward_kernel(const unsigned char* __restrict__ net, long long n,
                                                                  const float* __restrict__ X, float* __restrict__ Y,
                                                                  const R* __restrict__ d, const int* __restrict__ nbr,
                                                                  R* __restrict__ x, int accumulate, unsigned* status) {
  if (!wait_previous()) return;
  extern __shared__ __align__(128) unsigned char sm[];
  __shared__ uint64_t bar;
  start_weights(sm, net, &bar);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  const long long ra = (long long)blockIdx.x * kRows + warp * 16 + g, rb = ra + 8;
  const bool va = ra < n, vb = rb < n;
  uint32_t a1[7][4];
  R sa = R(0), sb = R(0);  // output scales (COARSE)
  if constexpr (MODE == kModeFeat) {
#pragma unroll
    for (int kk = 0; kk < 7; ++kk) {
      float2 p0 = make_float2(0.f, 0.f), p1 = p0, p2 = p0, p3 = p0;
      if (va) {
        p0 = *reinterpret_cast<const float2*>(X + ra * kIn + 16 * kk + 2 * t);
        p2 = *reinterpret_cast<const float2*>(X + ra * kIn + 16 * kk + 8 + 2 * t);
      }
      if (vb) {
        p1 = *reinterpret_cast<const float2*>(X + rb * kIn + 16 * kk + 2 * t);
        p3 = *reinterpret_cast<const float2*>(X + rb * kIn + 16 * kk + 8 + 2 * t);
      }
      a1[kk][0] = pack2(p0.x, p0.y);
      a1[kk][1] = pack2(p1.x, p1.y);
      a1[kk][2] = pack2(p2.x, p2.y);
      a1[kk][3] = pack2(p3.x, p3.y);
    }
  } else {
    int ea[7], eb[7];
    ea[0] = va ? (int)ra : 0;
    eb[0] = vb ? (int)rb : 0;
#pragma unroll
    for (int f = 0; f < 6; ++f) {
      ea[f + 1] = va ? nbr[ra * 6 + f] : 0;
      eb[f + 1] = vb ? nbr[rb * 6 + f] : 0;
    }
    // pass 1: squared norms of the 112 features of rows a and b (4 lanes per row)
    R qa = R(0), qb = R(0);
#pragma unroll
    for (int kk = 0; kk < 7; ++kk) {
      if (va && ea[kk] >= 0) {  // a missing neighbour (wall) contributes zero features
        const R* p = d + (size_t)ea[kk] * 16;
        const R u0 = p[2 * t], u1 = p[2 * t + 1], u2 = p[8 + 2 * t], u3 = p[9 + 2 * t];
        qa += u0 * u0 + u1 * u1 + u2 * u2 + u3 * u3;
      }
      if (vb && eb[kk] >= 0) {
        const R* p = d + (size_t)eb[kk] * 16;
        const R u0 = p[2 * t], u1 = p[2 * t + 1], u2 = p[8 + 2 * t], u3 = p[9 + 2 * t];
        qb += u0 * u0 + u1 * u1 + u2 * u2 + u3 * u3;
      }
    }
    qa += __shfl_xor_sync(0xffffffffu, qa, 1);
    qa += __shfl_xor_sync(0xffffffffu, qa, 2);
    qb += __shfl_xor_sync(0xffffffffu, qb, 1);
    qb += __shfl_xor_sync(0xffffffffu, qb, 2);
    sa = sqrt(qa);
    sb = sqrt(qb);
    const R ia = sa > R(0) ? R(1) / sa : R(0), ib = sb > R(0) ? R(1) / sb : R(0);
    // pass 2: normalised features -> BF16 A fragments (k-step kk = neighbour slot kk)
#pragma unroll
    for (int kk = 0; kk < 7; ++kk) {
      float f0 = 0.f, f1 = 0.f, f2 = 0.f, f3 = 0.f, h0 = 0.f, h1 = 0.f, h2 = 0.f, h3 = 0.f;
      if (va && ea[kk] >= 0) {
        const R* p = d + (size_t)ea[kk] * 16;
        f0 = (float)(p[2 * t] * ia); f1 = (float)(p[2 * t + 1] * ia);
        f2 = (float)(p[8 + 2 * t] * ia); f3 = (float)(p[9 + 2 * t] * ia);
      }
      if (vb && eb[kk] >= 0) {
        const R* p = d + (size_t)eb[kk] * 16;
        h0 = (float)(p[2 * t] * ib); h1 = (float)(p[2 * t + 1] * ib);
        h2 = (float)(p[8 + 2 * t] * ib); h3 = (float)(p[9 + 2 * t] * ib);
      }
      a1[kk][0] = pack2(f0, f1);
      a1[kk][1] = pack2(h0, h1);
      a1[kk][2] = pack2(f2, f3);
      a1[kk][3] = pack2(h2, h3);
    }
  }
  if (!mbar_wait(&bar, 0)) {
    // give up: report, and let the weights' copy land (a second bounded wait) before leaving,
    // so that it cannot write this CTA's shared memory after the CTA exits
    if (lane == 0) {
      atomicOr(status, DG_STATUS_WAIT);
      mbar_wait(&bar, 0);
    }
    __syncwarp();
    return;
  }
  float acc[16][4], out[2][4];
  layer1(sm, g, t, a1, acc);
  mlp_tail(sm, g, t, acc, out);
#pragma unroll
  for (int j = 0; j < 2; ++j) {
    const int c = 8 * j + 2 * t;
    if constexpr (MODE == kModeFeat) {
      if (va) *reinterpret_cast<float2*>(Y + ra * kOut + c) = make_float2(out[j][0], out[j][1]);
      if (vb) *reinterpret_cast<float2*>(Y + rb * kOut + c) = make_float2(out[j][2], out[j][3]);
    } else {
      R* pa = x + ra * kOut + c;
      R* pb = x + rb * kOut + c;
      if (va) { pa[0] = (accumulate ? pa[0] : R(0)) + sa * (R)out[j][0]; pa[1] = (accumulate ? pa[1] : R(0)) + sa * (R)out[j][1]; }
      if (vb) { pb[0] = (accumulate ? pb[0] : R(0)) + sb * (R)out[j][2]; pb[1] = (accumulate ? pb[1] : R(0)) + sb * (R)out[j][3]; }
    }
  }
}

// -------------------------------------------------------------- training
// One CTA: forward and backward of 128 samples, then its share of the weight gradient
// dW = dZ^T H (a contraction over its samples) on the tensor cores, written as one
// partial row; grad_reduce_kernel sums the rows in a fixed order.
//
// Latency and issue bound it (the arithmetic of 16384 samples is 2.8 GFMA, the data 8.4 MB):
// GELU and its derivative cost about as many issue slots as everything else, and one warp's
// chain of layers is serial. So a CTA has 16 warps, each with a 32 x 32 tile of every
// 128-wide layer: the four warps of a 32-sample stripe exchange activations through shared
// memory under a barrier of their own, so that stripes drift apart and one's matrix products
// run beside another's GELU. Every tile is kept sample-major and read by ldmatrix, transposed
// where the samples are the contraction, and the 16384 samples are one wave of 128 CTAs.
// gelu' stays in registers. With four warps per CTA, each with 16 samples and all columns,
// feature-major copies by 2-byte stores and 64 samples per CTA (1.7 waves):
// 63 us at 16384 samples; now 19 us.
constexpr int kTRows = 128, kTWarps = 16, kStripes = 4, kLdY = 24;
constexpr int sX = kPBytes;
constexpr int sH1 = sX + kTRows * kLd1 * 2;
constexpr int sH2 = sH1 + kTRows * kLd2 * 2;
constexpr int sDZ2 = sH2 + kTRows * kLd2 * 2;
constexpr int sDY = sDZ2 + kTRows * kLd2 * 2;
constexpr int sDZ1 = kPW2;                       // takes the place of W2 once dH1 has been formed
constexpr int sBsum = sDY + kTRows * kLdY * 2;   // [stripe][128 + 128 + 16] column sums of dZ1, dZ2, dY
constexpr int sLoss = sBsum + kStripes * (2 * kHid + kOut) * 4;
constexpr int sRow = sLoss + kTWarps * 4;        // the pair each sample slot holds, -1 past the batch
constexpr int kTrainSmem = sRow + kTRows * 8;
constexpr int kPartLd = kNP + 16;                // partial row: gradient, then the loss sum
static_assert(kTrainSmem <= 227 * 1024, "training tile exceeds shared memory");
static_assert(sX % 16 == 0 && sH1 % 16 == 0 && sDY % 16 == 0 && sBsum % 16 == 0 && sRow % 8 == 0, "alignment");
static_assert(kHid * kLd2 >= kTRows * kLd2, "dZ1 fits in the place of W2");
static_assert(kPartLd % 4 == 0 && kPBytes % 16 == 0, "partial rows are read by 16 bytes");

__device__ __forceinline__ long long sample_row(long long seed, long long step, long long s, long long npairs) {
  if (seed < 0) return s;
  unsigned long long z = (unsigned long long)seed * 0x9E3779B97F4A7C15ull +
                         (unsigned long long)step * 0xD1B54A32D192ED03ull + (unsigned long long)s * 0x8CB92BA72F3D8DD7ull;
  z ^= z >> 30;
  z *= 0xBF58476D1CE4E5B9ull;
  z ^= z >> 27;
  z *= 0x94D049BB133111EBull;
  z ^= z >> 31;
  return (long long)(z % (unsigned long long)npairs);
}

// four 8 x 8 BF16 matrices, one row address per lane; trans: each is transposed on the way
template <bool TRANS>
__device__ __forceinline__ void ldmatrix4(uint32_t (&r)[4], const unsigned char* p) {
  const uint32_t a = static_cast<uint32_t>(__cvta_generic_to_shared(p));
  if constexpr (TRANS)
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(a) : "memory");
  else
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(a) : "memory");
}

// acc[mt][nt] += A B over KS steps of 16 for a (16 MT) x (8 NT) tile at (m0, n0).
// A: [m][k] in shared memory, or [k][m] with TA; B: [n][k], or [k][n] with TB; LDA, LDB the
// row lengths. With TA or TB the matrix loads transpose.
template <int MT, int NT, int KS, bool TA, bool TB, int LDA, int LDB>
__device__ __forceinline__ void tile_mma(const unsigned char* A, const unsigned char* B, int m0, int n0, int lane,
                                         float (&acc)[MT][NT][4]) {
  static_assert(NT % 2 == 0, "B is loaded two column groups at a time");
  const int lo = lane & 7, q = (lane >> 3) & 1, hi = lane >> 4;
  const unsigned char* pa = A + 2 * (TA ? (lo + 8 * hi) * LDA + m0 + 8 * q : (m0 + lo + 8 * q) * LDA + 8 * hi);
  const unsigned char* pb = B + 2 * (TB ? (lo + 8 * q) * LDB + n0 + 8 * hi : (n0 + lo + 8 * hi) * LDB + 8 * q);
#pragma unroll
  for (int k = 0; k < KS; ++k) {
    uint32_t a[MT][4], b[NT / 2][4];
#pragma unroll
    for (int m = 0; m < MT; ++m) ldmatrix4<TA>(a[m], pa + 2 * (TA ? 16 * k * LDA + 16 * m : 16 * m * LDA + 16 * k));
#pragma unroll
    for (int n = 0; n < NT / 2; ++n) ldmatrix4<TB>(b[n], pb + 2 * (TB ? 16 * k * LDB + 16 * n : 16 * n * LDB + 16 * k));
#pragma unroll
    for (int m = 0; m < MT; ++m)
#pragma unroll
      for (int n = 0; n < NT; ++n) mma16816(acc[m][n], a[m], b[n >> 1][2 * (n & 1)], b[n >> 1][2 * (n & 1) + 1]);
  }
}

template <int MT, int NT>
__device__ __forceinline__ void zero_tile(float (&acc)[MT][NT][4]) {
#pragma unroll
  for (int m = 0; m < MT; ++m)
#pragma unroll
    for (int n = 0; n < NT; ++n) acc[m][n][0] = acc[m][n][1] = acc[m][n][2] = acc[m][n][3] = 0.f;
}

// a tile as BF16 into a sample-major array [sample][LD] at (m0, n0)
template <int MT, int NT, int LD>
__device__ __forceinline__ void put_tile(unsigned char* dst, int m0, int n0, int g, int t,
                                         const float (&v)[MT][NT][4]) {
#pragma unroll
  for (int m = 0; m < MT; ++m)
#pragma unroll
    for (int n = 0; n < NT; ++n) {
      unsigned char* p = dst + 2 * ((m0 + 16 * m + g) * LD + n0 + 8 * n + 2 * t);
      *reinterpret_cast<uint32_t*>(p) = pack2(v[m][n][0], v[m][n][1]);
      *reinterpret_cast<uint32_t*>(p + 16 * LD) = pack2(v[m][n][2], v[m][n][3]);
    }
}

// a tile in FP32 into the row-major matrix dst [.][ld] at (m0, n0)
template <int MT, int NT>
__device__ __forceinline__ void put_grad(float* dst, int ld, int m0, int n0, int g, int t,
                                         const float (&v)[MT][NT][4]) {
#pragma unroll
  for (int m = 0; m < MT; ++m)
#pragma unroll
    for (int n = 0; n < NT; ++n) {
      float* p = dst + (m0 + 16 * m + g) * ld + n0 + 8 * n + 2 * t;
      *reinterpret_cast<float2*>(p) = make_float2(v[m][n][0], v[m][n][1]);
      *reinterpret_cast<float2*>(p + 8 * ld) = make_float2(v[m][n][2], v[m][n][3]);
    }
}

// column sums over the rows of a tile -> dst[8 n + .]
template <int MT, int NT>
__device__ __forceinline__ void tile_colsum(const float (&v)[MT][NT][4], float* dst, int lane) {
#pragma unroll
  for (int n = 0; n < NT; ++n) {
    float c0 = 0.f, c1 = 0.f;
#pragma unroll
    for (int m = 0; m < MT; ++m) {
      c0 += v[m][n][0] + v[m][n][2];
      c1 += v[m][n][1] + v[m][n][3];
    }
#pragma unroll
    for (int o = 4; o < 32; o <<= 1) {
      c0 += __shfl_xor_sync(0xffffffffu, c0, o);
      c1 += __shfl_xor_sync(0xffffffffu, c1, o);
    }
    if (lane < 4) {
      dst[8 * n + 2 * lane] = c0;
      dst[8 * n + 2 * lane + 1] = c1;
    }
  }
}

// acc = bias, per column
template <int MT, int NT>
__device__ __forceinline__ void bias_tile(const float* b, int n0, int t, float (&acc)[MT][NT][4]) {
#pragma unroll
  for (int n = 0; n < NT; ++n) {
    const float2 bb = *reinterpret_cast<const float2*>(b + n0 + 8 * n + 2 * t);
#pragma unroll
    for (int m = 0; m < MT; ++m) {
      acc[m][n][0] = acc[m][n][2] = bb.x;
      acc[m][n][1] = acc[m][n][3] = bb.y;
    }
  }
}

// z -> gelu(z) in place; gelu'(z) as packed BF16
__device__ __forceinline__ void gelu_tile(float (&z)[2][4][4], uint32_t (&d)[2][4][2]) {
#pragma unroll
  for (int m = 0; m < 2; ++m)
#pragma unroll
    for (int n = 0; n < 4; ++n)
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const float z0 = z[m][n][2 * q], z1 = z[m][n][2 * q + 1];
        d[m][n][q] = pack2(gelu_d(z0), gelu_d(z1));
        z[m][n][2 * q] = gelu(z0);
        z[m][n][2 * q + 1] = gelu(z1);
      }
}

__device__ __forceinline__ void scale_tile(float (&v)[2][4][4], const uint32_t (&d)[2][4][2]) {
#pragma unroll
  for (int m = 0; m < 2; ++m)
#pragma unroll
    for (int n = 0; n < 4; ++n)
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        v[m][n][2 * q] *= bf16_to_f(d[m][n][q] & 0xffff);
        v[m][n][2 * q + 1] *= bf16_to_f(d[m][n][q] >> 16);
      }
}

// the 128 threads of one 32-sample stripe
__device__ __forceinline__ void stripe_sync(int stripe) {
  asm volatile("bar.sync %0, %1;" ::"r"(stripe + 1), "r"(32 * kTWarps / kStripes) : "memory");
}

__global__ void __launch_bounds__(32 * kTWarps, 1) mlp_grad_kernel(const unsigned char* __restrict__ net,
                                                                  const float* __restrict__ X,
                                                                  const float* __restrict__ T, long long npairs,
                                                                  int batch, long long seed, long long step,
                                                                  float* __restrict__ part, unsigned* status) {
  if (!wait_previous()) return;
  extern __shared__ __align__(128) unsigned char sm[];
  __shared__ uint64_t bar;
  __shared__ int ok_all;
  long long* row = reinterpret_cast<long long*>(sm + sRow);
  if (threadIdx.x < kTRows) {
    const long long s = (long long)blockIdx.x * kTRows + threadIdx.x;
    row[threadIdx.x] = s < batch ? sample_row(seed, step, s, npairs) : -1;
  }
  if (threadIdx.x == 0) ok_all = 1;
  start_weights(sm, net, &bar);  // its barrier also orders row[] and ok_all
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  const int stripe = warp / (kTWarps / kStripes), wc = warp % (kTWarps / kStripes);
  const int m0 = 32 * stripe, n0 = 32 * wc;
  {
    // the samples' features, BF16: 28 groups of four per row
    constexpr int kC4 = kIn / 4, kN = kTRows * kC4 / (32 * kTWarps);
    static_assert(kTRows * kC4 % (32 * kTWarps) == 0, "whole groups per thread");
    float4 v[kN];
#pragma unroll
    for (int i = 0; i < kN; ++i) {
      const int c = threadIdx.x + i * 32 * kTWarps;
      const long long r = row[c / kC4];
      v[i] = r >= 0 ? *reinterpret_cast<const float4*>(X + r * kIn + 4 * (c % kC4)) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
#pragma unroll
    for (int i = 0; i < kN; ++i) {
      const int c = threadIdx.x + i * 32 * kTWarps;
      *reinterpret_cast<uint2*>(sm + sX + 2 * ((c / kC4) * kLd1 + 4 * (c % kC4))) =
          make_uint2(pack2(v[i].x, v[i].y), pack2(v[i].z, v[i].w));
    }
  }
  if (!mbar_wait(&bar, 0)) ok_all = 0;
  __syncthreads();
  if (!ok_all) {
    if (threadIdx.x == 0) {  // report; the copy in flight lands before the CTA leaves
      atomicOr(status, DG_STATUS_WAIT);
      mbar_wait(&bar, 0);
    }
    __syncthreads();
    return;
  }
  const float* Bs = reinterpret_cast<const float*>(sm + kPB);
  float* bsum = reinterpret_cast<float*>(sm + sBsum) + stripe * (2 * kHid + kOut);
  float acc[2][4][4];
  uint32_t G1[2][4][2], G2[2][4][2];
  // ---- forward
  bias_tile<2, 4>(Bs, n0, t, acc);
  tile_mma<2, 4, kIn / 16, false, false, kLd1, kLd1>(sm + sX, sm + kPW1, m0, n0, lane, acc);
  gelu_tile(acc, G1);
  put_tile<2, 4, kLd2>(sm + sH1, m0, n0, g, t, acc);
  stripe_sync(stripe);
  bias_tile<2, 4>(Bs + kHid, n0, t, acc);
  tile_mma<2, 4, kHid / 16, false, false, kLd2, kLd2>(sm + sH1, sm + kPW2, m0, n0, lane, acc);
  gelu_tile(acc, G2);
  put_tile<2, 4, kLd2>(sm + sH2, m0, n0, g, t, acc);
  stripe_sync(stripe);
  // ---- layer 3 and the loss: warps 0 and 1 of the stripe take 16 samples and all 16 outputs each
  float lsum = 0.f;
  if (wc < 2) {
    float out[1][2][4];
    const int mb = m0 + 16 * wc;
    bias_tile<1, 2>(Bs + 2 * kHid, 0, t, out);
    tile_mma<1, 2, kHid / 16, false, false, kLd2, kLd2>(sm + sH2, sm + kPW3, mb, 0, lane, out);
    const float sc = 2.0f / (float)batch;
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const long long r = row[mb + g + 8 * q];
#pragma unroll
      for (int n = 0; n < 2; ++n) {
        const float2 y = r >= 0 ? *reinterpret_cast<const float2*>(T + r * kOut + 8 * n + 2 * t) : make_float2(0.f, 0.f);
        const float r0 = r >= 0 ? out[0][n][2 * q] - y.x : 0.f, r1 = r >= 0 ? out[0][n][2 * q + 1] - y.y : 0.f;
        lsum += r0 * r0 + r1 * r1;
        out[0][n][2 * q] = sc * r0;  // dY
        out[0][n][2 * q + 1] = sc * r1;
      }
    }
    put_tile<1, 2, kLdY>(sm + sDY, mb, 0, g, t, out);
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) lsum += __shfl_xor_sync(0xffffffffu, lsum, o);
    // the stripe's column sums of dY: both halves' below, each from its own 16-column slot
    tile_colsum<1, 2>(out, bsum + (wc ? kHid : 0), lane);
  }
  if (lane == 0) reinterpret_cast<float*>(sm + sLoss)[warp] = lsum;
  stripe_sync(stripe);
  if (wc == 0 && lane < kOut) bsum[2 * kHid + lane] = bsum[lane] + bsum[kHid + lane];
  stripe_sync(stripe);
  // ---- dH2 = dY W3, dZ2 = dH2 . gelu'(Z2)
  zero_tile<2, 4>(acc);
  tile_mma<2, 4, 1, false, true, kLdY, kLd2>(sm + sDY, sm + kPW3, m0, n0, lane, acc);
  scale_tile(acc, G2);
  tile_colsum<2, 4>(acc, bsum + kHid + n0, lane);
  put_tile<2, 4, kLd2>(sm + sDZ2, m0, n0, g, t, acc);
  stripe_sync(stripe);
  // ---- dH1 = dZ2 W2, dZ1 = dH1 . gelu'(Z1)
  zero_tile<2, 4>(acc);
  tile_mma<2, 4, kHid / 16, false, true, kLd2, kLd2>(sm + sDZ2, sm + kPW2, m0, n0, lane, acc);
  scale_tile(acc, G1);
  tile_colsum<2, 4>(acc, bsum + n0, lane);
  __syncthreads();  // every stripe is through with W2
  put_tile<2, 4, kLd2>(sm + sDZ1, m0, n0, g, t, acc);
  __syncthreads();
  // ---- weight gradients of this CTA: dW1 = dZ1^T X, dW2 = dZ2^T H1, dW3 = dY^T H2
  float* P = part + (size_t)blockIdx.x * kPartLd;
  zero_tile<2, 4>(acc);
  tile_mma<2, 4, kTRows / 16, true, true, kLd2, kLd2>(sm + sDZ2, sm + sH1, m0, n0, lane, acc);
  put_grad<2, 4>(P + oW2, kHid, m0, n0, g, t, acc);
  zero_tile<2, 4>(acc);
  static_assert(kIn == 3 * 32 + 16, "three warps with 32 columns of dW1 and one with 16");
  if (wc < 3) {
    tile_mma<2, 4, kTRows / 16, true, true, kLd2, kLd1>(sm + sDZ1, sm + sX, m0, n0, lane, acc);
    put_grad<2, 4>(P + oW1, kIn, m0, n0, g, t, acc);
  } else {
    float last[2][2][4], w3[1][4][4];
    zero_tile<2, 2>(last);
    tile_mma<2, 2, kTRows / 16, true, true, kLd2, kLd1>(sm + sDZ1, sm + sX, m0, n0, lane, last);
    put_grad<2, 2>(P + oW1, kIn, m0, n0, g, t, last);
    zero_tile<1, 4>(w3);
    tile_mma<1, 4, kTRows / 16, true, true, kLdY, kLd2>(sm + sDY, sm + sH2, 0, m0, lane, w3);
    put_grad<1, 4>(P + oW3, kHid, 0, m0, g, t, w3);
  }
  // bias gradients and the loss: sums over the stripes or warps in a fixed order
  const float* bs = reinterpret_cast<const float*>(sm + sBsum);
  for (int i = threadIdx.x; i < 2 * kHid + kOut; i += blockDim.x) {
    float s = 0.f;
    for (int w = 0; w < kStripes; ++w) s += bs[w * (2 * kHid + kOut) + i];
    const int dst = i < kHid ? ob1 + i : i < 2 * kHid ? ob2 + (i - kHid) : ob3 + (i - 2 * kHid);
    P[dst] = s;
  }
  if (threadIdx.x == 0) {
    const float* ls = reinterpret_cast<const float*>(sm + sLoss);
    float s = 0.f;
    for (int w = 0; w < kTWarps; ++w) s += ls[w];
    P[kNP] = s;
  }
}

// grad[p] = sum_c part[c][p]; loss = sum_c part[c][kNP] / batch (fixed order). Bound by the
// latency of its loads: 16 bytes of four consecutive entries per thread, eight threads per
// group with every eighth partial row each, their sums joined in shared memory. One thread
// per entry over all rows: 8.2 us for 16384 samples (256 rows), now 3.5 us (128 rows).
constexpr int kRedCols = 32, kRedRows = 8;
__global__ void __launch_bounds__(kRedCols* kRedRows) grad_reduce_kernel(const float* __restrict__ part, int nparts,
                                                                         int batch, float* __restrict__ grad,
                                                                         float* __restrict__ loss) {
  if (!wait_previous()) return;
  __shared__ float4 sum[kRedRows][kRedCols];
  const int x = threadIdx.x % kRedCols, y = threadIdx.x / kRedCols;
  const int q = blockIdx.x * kRedCols + x;  // group of four entries
  float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
  if (4 * q <= kNP) {
    const float4* p = reinterpret_cast<const float4*>(part) + q;
#pragma unroll 8
    for (int c = y; c < nparts; c += kRedRows) {
      const float4 v = p[(size_t)c * (kPartLd / 4)];
      s.x += v.x; s.y += v.y; s.z += v.z; s.w += v.w;
    }
  }
  sum[y][x] = s;
  __syncthreads();
  if (threadIdx.x >= 4 * kRedCols) return;
  const int p = 4 * blockIdx.x * kRedCols + threadIdx.x;
  if (p > kNP) return;
  float r = 0.f;
#pragma unroll
  for (int i = 0; i < kRedRows; ++i) r += reinterpret_cast<const float*>(sum[i])[threadIdx.x];
  if (p < kNP) grad[p] = r;
  else if (loss) *loss = r / (float)batch;
}

__global__ void adam_kernel(float* __restrict__ theta, const float* __restrict__ grad, float* __restrict__ m,
                            float* __restrict__ v, float lr_t, float b1, float b2, float eps, float bc2) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= kNP) return;
  const float gr = grad[p];
  const float mm = b1 * m[p] + (1.0f - b1) * gr;
  const float vv = b2 * v[p] + (1.0f - b2) * gr * gr;
  m[p] = mm;
  v[p] = vv;
  theta[p] -= lr_t * mm / (sqrtf(vv / bc2) + eps);
}

// Training pairs of the coarsest level: one thread per element.
__global__ void pairs_kernel(int ne, const double* __restrict__ d, const double* __restrict__ x,
                             const double* __restrict__ q, const int* __restrict__ nbr, float* __restrict__ X,
                             float* __restrict__ T, float* __restrict__ s) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= ne) return;
  int src[7];
  src[0] = e;
  for (int f = 0; f < 6; ++f) src[f + 1] = nbr[(size_t)e * 6 + f];
  double ss = 0.0;
  for (int k = 0; k < 7; ++k)
    for (int i = 0; i < 16; ++i) {
      const double u = src[k] >= 0 ? d[(size_t)src[k] * 16 + i] : 0.0;  // zero across a wall
      ss += u * u;
    }
  const double nrm = sqrt(ss);
  const double inv = nrm > 0.0 ? 1.0 / nrm : 0.0;
  for (int k = 0; k < 7; ++k)
    for (int i = 0; i < 16; ++i)
      X[(size_t)e * kIn + 16 * k + i] = src[k] >= 0 ? (float)(d[(size_t)src[k] * 16 + i] * inv) : 0.0f;
  for (int i = 0; i < 16; ++i)
    T[(size_t)e * kOut + i] = (float)(x[(size_t)e * 16 + i] * inv + (q ? nrm * q[(size_t)e * 16 + i] : 0.0));
  s[e] = (float)nrm;
}

// opt-in, once per kernel, to more than 48 KB of dynamic shared memory
std::mutex g_optin_mu;
std::vector<const void*> g_optin_done;
template <class K>
int smem_opt_in(K kernel, int bytes) {
  std::lock_guard<std::mutex> lock(g_optin_mu);
  const void* key = reinterpret_cast<const void*>(kernel);
  for (const void* k : g_optin_done)
    if (k == key) return 0;
  if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes) != cudaSuccess) return 1;
  g_optin_done.push_back(key);
  return 0;
}

long long grad_parts(long long batch) { return (batch + kTRows - 1) / kTRows; }

bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

// status word of the handle-less calls
__device__ unsigned g_mlp_status;

unsigned* mlp_status_ptr() {
  static std::mutex mu;
  static unsigned* p = nullptr;
  std::lock_guard<std::mutex> lock(mu);
  if (!p) {
    void* a = nullptr;
    if (cudaGetSymbolAddress(&a, g_mlp_status) != cudaSuccess) return nullptr;
    p = static_cast<unsigned*>(a);
  }
  return p;
}

}  // namespace

int net_bytes() { return kPBytes; }

template <class R>
int learned_coarse(Handle* h, const R* g, R* x, bool accumulate, cudaStream_t st) {
  if (!h->net_ready) return fail(h, DG_ERR_STATE, "no coarse network set (dg_set_coarse_network)");
  const Level& C = h->lev[h->nlev - 1];
  if (C.k != 1) return fail(h, DG_ERR_ARG, "the learned coarse correction needs k = 1 on the coarsest level");
  if (smem_opt_in(mlp_forward_kernel<kModeCoarse, R>, kPBytes))
    return fail(h, DG_ERR_CUDA, "cannot opt in to the shared memory of the network kernel");
  const int grid = (int)((h->ne + kRows - 1) / kRows);
  launch(mlp_forward_kernel<kModeCoarse, R>, grid, 32 * kWarps, kPBytes, st, h->net, h->ne, nullptr, nullptr, g,
         h->nbr, x, accumulate ? 1 : 0, h->status);
  DG_LAUNCH_CHECK(h);
  return DG_OK;
}
template int learned_coarse<double>(Handle*, const double*, double*, bool, cudaStream_t);
template int learned_coarse<float>(Handle*, const float*, float*, bool, cudaStream_t);

}  // namespace dg

using namespace dg;

#define MLP_CUDA(call)                                                                      \
  do {                                                                                      \
    cudaError_t e_ = (call);                                                                \
    if (e_ != cudaSuccess) return fail(nullptr, DG_ERR_CUDA, std::string(#call) + ": " + cudaGetErrorString(e_)); \
  } while (0)

extern "C" {

long long dg_mlp_workspace_bytes(long long rows) {
  if (rows < 1) rows = 1;
  return (long long)kPBytes + grad_parts(rows) * (long long)kPartLd * 4;
}

int dg_mlp_forward(const float* theta, const float* X, long long n, float* Y, void* ws, void* stream) {
  if (!theta || !X || !Y || !ws || n < 0) return fail(nullptr, DG_ERR_ARG, "dg_mlp_forward: bad argument");
  if (!aligned16(ws) || !aligned16(X) || !aligned16(Y)) return fail(nullptr, DG_ERR_ARG, "dg_mlp_forward: unaligned");
  if (n == 0) return DG_OK;
  cudaStream_t st = as_stream(stream);
  unsigned* status = mlp_status_ptr();
  if (!status) return fail(nullptr, DG_ERR_CUDA, "cannot look up the status word");
  unsigned char* net = static_cast<unsigned char*>(ws);
  launch(pack_kernel, (kPackSlots + 255) / 256, 256, 0, st, theta, net);
  MLP_CUDA(cudaGetLastError());
  if (smem_opt_in(mlp_forward_kernel<kModeFeat, float>, kPBytes))
    return fail(nullptr, DG_ERR_CUDA, "cannot opt in to the shared memory of the network kernel");
  const long long grid = (n + kRows - 1) / kRows;
  if (grid > 0x7fffffffLL) return fail(nullptr, DG_ERR_ARG, "dg_mlp_forward: too many rows");
  launch(mlp_forward_kernel<kModeFeat, float>, (unsigned)grid, 32 * kWarps, kPBytes, st, net, n, X, Y, nullptr,
         nullptr, nullptr, 0, status);
  MLP_CUDA(cudaGetLastError());
  return DG_OK;
}

int dg_mlp_grad(const float* theta, const float* X, const float* T, long long npairs, int batch, long long seed,
                long long step, float* grad, float* loss, void* ws, void* stream) {
  if (!theta || !X || !T || !grad || !ws || batch < 1 || npairs < 1)
    return fail(nullptr, DG_ERR_ARG, "dg_mlp_grad: bad argument");
  if (seed < 0 && batch > npairs) return fail(nullptr, DG_ERR_ARG, "dg_mlp_grad: batch > npairs without sampling");
  if (!aligned16(ws) || !aligned16(X) || !aligned16(T)) return fail(nullptr, DG_ERR_ARG, "dg_mlp_grad: unaligned");
  cudaStream_t st = as_stream(stream);
  unsigned* status = mlp_status_ptr();
  if (!status) return fail(nullptr, DG_ERR_CUDA, "cannot look up the status word");
  unsigned char* net = static_cast<unsigned char*>(ws);
  float* part = reinterpret_cast<float*>(net + kPBytes);
  launch(pack_kernel, (kPackSlots + 255) / 256, 256, 0, st, theta, net);
  MLP_CUDA(cudaGetLastError());
  if (smem_opt_in(mlp_grad_kernel, kTrainSmem))
    return fail(nullptr, DG_ERR_CUDA, "cannot opt in to the shared memory of the training kernel");
  const int nparts = (int)grad_parts(batch);
  launch(mlp_grad_kernel, nparts, 32 * kTWarps, kTrainSmem, st, net, X, T, npairs, batch, seed, step, part, status);
  MLP_CUDA(cudaGetLastError());
  launch(grad_reduce_kernel, (kNP + 4 * kRedCols) / (4 * kRedCols), kRedCols * kRedRows, 0, st, part, nparts, batch,
         grad, loss);
  MLP_CUDA(cudaGetLastError());
  return DG_OK;
}

int dg_mlp_adam(float* theta, const float* grad, float* m, float* v, long long t, double lr, double beta1, double beta2,
                double eps, void* stream) {
  if (!theta || !grad || !m || !v || t < 1 || !(lr > 0.0) || !(beta1 >= 0.0 && beta1 < 1.0) ||
      !(beta2 >= 0.0 && beta2 < 1.0) || !(eps > 0.0))
    return fail(nullptr, DG_ERR_ARG, "dg_mlp_adam: bad argument");
  const double bc1 = 1.0 - std::pow(beta1, (double)t), bc2 = 1.0 - std::pow(beta2, (double)t);
  adam_kernel<<<(kNP + 255) / 256, 256, 0, as_stream(stream)>>>(theta, grad, m, v, (float)(lr / bc1), (float)beta1,
                                                                 (float)beta2, (float)eps, (float)bc2);
  MLP_CUDA(cudaGetLastError());
  return DG_OK;
}

int dg_set_coarse_network(dg_handle* hh, const float* theta, void* stream) {
  Handle* h = reinterpret_cast<Handle*>(hh);
  if (!h) return DG_ERR_ARG;
  if (!theta) {
    h->net_ready = false;
    return DG_OK;
  }
  if (h->lev[h->nlev - 1].k != 1)
    return fail(h, DG_ERR_ARG, "the learned coarse correction needs k = 1 on the coarsest level");
  if (!h->net) DG_CUDA(h, cudaMalloc((void**)&h->net, kPBytes));
  launch(pack_kernel, (kPackSlots + 255) / 256, 256, 0, as_stream(stream), theta, h->net);
  DG_LAUNCH_CHECK(h);
  h->net_ready = true;
  return DG_OK;
}

int dg_coarse_pairs(dg_handle* hh, const double* d, const double* x, const double* q, float* X, float* T, float* s,
                    void* stream) {
  Handle* h = reinterpret_cast<Handle*>(hh);
  if (!h) return DG_ERR_ARG;
  if (!d || !x || !X || !T || !s) return fail(h, DG_ERR_ARG, "dg_coarse_pairs: null pointer");
  if (h->lev[h->nlev - 1].k != 1) return fail(h, DG_ERR_ARG, "dg_coarse_pairs needs k = 1 on the coarsest level");
  pairs_kernel<<<(h->ne + 127) / 128, 128, 0, as_stream(stream)>>>(h->ne, d, x, q, h->nbr, X, T, s);
  DG_LAUNCH_CHECK(h);
  return DG_OK;
}

int dg_record_coarse(dg_handle* hh, double* buf, int capacity) {
  Handle* h = reinterpret_cast<Handle*>(hh);
  if (!h) return DG_ERR_ARG;
  if (buf && capacity < 1) return fail(h, DG_ERR_ARG, "dg_record_coarse: capacity must be >= 1");
  h->rec_buf = buf;
  h->rec_cap = buf ? capacity : 0;
  h->rec_count = 0;
  return DG_OK;
}

int dg_recorded(const dg_handle* hh, int* count) {
  const Handle* h = reinterpret_cast<const Handle*>(hh);
  if (!h || !count) return DG_ERR_ARG;
  *count = h->rec_count;
  return DG_OK;
}

}  // extern "C"
