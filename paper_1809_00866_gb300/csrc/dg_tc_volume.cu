// Tensor-core volume pass of the FP32 preconditioner cycle's Jacobian action (sm_103a).
//
// The convective volume term of the linearised residual (Eq. (jacTrilFnotNU): the quadrature of
// d(u (x) u)[du] : grad phi_j in Eq. (NSdiscrRes)) needs the velocity variation at the Gauss
// points and the integral of the weighted products against the basis. Here both contractions run
// as dense per-element GEMMs on the 5th-generation tensor cores (tcgen05.mma, kind::f16: FP16 or
// BF16 operands, FP32 accumulation in tensor memory), 8 elements per tile:
//
//   interpolation  D1[q][(e,f)] = sum_m L_m(x_q) * sigma_e c_{e,f,m}
//                  M = 128 Gauss points (125 used), N = 32 (24 = 8 x 3 velocity components),
//                  K = 48 modes (35 used);
//   integration    D2[(e,s)][m] = sum_q P_{e,s}(x_q) * W_m L_m(x_q)
//                  M = 128 (48 = 8 x 6 symmetric products), N = 32 modes (the 20 of degree <= k-1
//                  that the derivative of a test function meets), K = 128 points,
//
// with L_m the plain Legendre products and c their coefficients (dg_pencil.h), W_m the factors that
// make coefficients of the integrals, and P_{e,s}(x_q) = w_q (u_p ub_i + ub_p u_i) scaled by sigma_e
// tau_e. The scales are powers of two per element: sigma_e from the largest velocity coefficient of
// the tile's input and tau_e from the largest linearisation velocity at the element's points
// (computed once per linearisation), so that every 16-bit operand lies near unit size whatever the
// magnitude of the Krylov vector the cycle is applied to. Power-of-two scales are exact, and the FP32
// results are unscaled exactly.
//
// Everything else is the FP32 arithmetic of the volume pass (dg_volume_phases.h): corrected gradients
// with the BR2 liftings, the viscous flux, the pressure and continuity terms as exact modal
// derivatives, the six face contributions and the mass shift (Eqs. (vflux), (massBil)).
//
// Bound: instruction issue and the per-tile chain (load, MMA, products, MMA, derivatives); the tensor
// pipe is under 1 % busy. So each phase is written for few instructions, the elements' rows are
// scaled, measured for sigma and converted to the operand while they are loaded, and four CTAs share an
// SM (tiles of 21 elements, which fill the MMAs' rows, left two CTAs waiting on each other's phases).
// At 32^3 P4: 127 us with those, 82 us now; at 24 x 12 x 12 P3 15 us (events included). The CUDA-core pass
// (dg_volume.cu) takes 68 and 12 us.
//
// Operand layout in shared memory (K-major, no swizzle): cores of 8 rows x 16 bytes; the shared
// memory descriptor's leading byte offset is the distance of K-adjacent cores, the stride byte
// offset that of row-adjacent 8-row groups. The 16-bit basis tables (D1's A operand, D2's B
// operand) are built on the host once per handle. The products' operand uses a K-core distance
// of 144 bytes, so that the 2-byte stores of 32 consecutive points hit 32 distinct banks.
//
// One elected thread issues the MMAs and commits them to an mbarrier; every wait is bounded
// (DG_STATUS_WAIT, then a second bounded wait for the MMAs in flight before the tensor memory is
// released).
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <vector>

#include "dg_async.h"
#include "dg_internal.h"
#include "dg_launch.h"
#include "dg_volume_phases.h"

namespace dg {
namespace {

constexpr int kTcE = 8;                 // elements per tile (6 x 8 = 48 rows of D2)
constexpr int kTcThreads = 256;         // warps w and w + 4 read TMEM lane quarter w % 4
constexpr unsigned kTcCols = 64;        // TMEM columns per CTA: D1 at 0..31, D2 at 32..63
constexpr unsigned kTcD2 = 32;
constexpr int kQP = 128;                // padded Gauss points
constexpr int kMP = 48;                 // padded modes of the interpolation
constexpr int kN1 = 32;                 // N of the interpolation
constexpr int kN2 = 32;                 // N of the integration: padded modes of degree <= k - 1
// Shared-memory byte offsets of the operands. The integration's A operand holds the 48 rows in use;
// the MMA's other 80 rows read the bytes after it (inside the CTA's own allocation) and give rows
// of D2 that nobody reads.
constexpr unsigned kA2 = 0;             // [48 (e,s)][128 q], K-cores 144 B apart
constexpr unsigned kA2Bytes = 6 * 16 * 144, kA2Read = 16 * 16 * 144;
constexpr unsigned kTA1 = kA2Bytes;     // [128 q][48 m]
constexpr unsigned kTB2 = kTA1 + 12288;  // [32 m][128 q]
constexpr unsigned kTabBytes = 20480;   // TA1 + TB2
constexpr unsigned kB1 = kTA1 + kTabBytes;  // [32 (e,f)][48 m]
constexpr unsigned kB1Bytes = 4 * 6 * 128;
constexpr unsigned kKc = 128, kKcA2 = 144;  // K-core distances
constexpr unsigned kRgTA1 = 6 * 128, kRgTB2 = 16 * 128, kRgB1 = 6 * 128, kRgA2 = 16 * 144;  // row-group distances

template <int K>
struct TcSz : VolPhases<K, float, kTcE> {
  using Ph = VolPhases<K, float, kTcE>;
  using Ph::GEO, Ph::LD, Ph::N1, Ph::NB, Ph::NBM, Ph::NQ, Ph::NT;
  static constexpr unsigned SC = kB1 + kB1Bytes;                                  // [4][NB] rows
  static constexpr unsigned ST = SC + ((4 * NB * LD * 4 + 127) / 128) * 128;     // [6][NBM] rows
  static constexpr unsigned GE = ST + ((6 * NT * LD * 4 + 127) / 128) * 128;     // [E][GEO]
  static constexpr unsigned SS = GE + kTcE * GEO * 4;                             // [2][NB] mode scales, inverses
  static constexpr unsigned FID = SS + 2 * NB * 4;                                // [E][6] face records
  static constexpr unsigned BYTES = FID + kTcE * 6 * 4;
  static_assert(kTcE == kFaceGroup, "a tile's own faces are three groups");
  static_assert(NQ <= kQP && NB <= kMP && NBM <= kN2 && BYTES >= kA2 + kA2Read, "tile sizes");
  // the gradient before the products are formed, the output after the integration
  static_assert(9 * NT * LD * 4 <= (int)kA2Bytes && 4 * NB * LD * 4 <= (int)kA2Bytes, "fit the products' buffer");
};

// byte offset of element (r, k) in a K-major no-swizzle operand
__host__ __device__ constexpr unsigned core_off(int r, int k, unsigned kcore, unsigned rgroup) {
  return (unsigned)(r / 8) * rgroup + (unsigned)(k / 8) * kcore + (unsigned)(r % 8) * 16 + (unsigned)(k % 8) * 2;
}

// ---------------------------------------------------------------- tcgen05 wrappers
__device__ __forceinline__ uint64_t umma_smem_desc(unsigned addr, unsigned kcore, unsigned rgroup) {
  uint64_t d = (uint64_t)((addr & 0x3FFFF) >> 4);
  d |= (uint64_t)((kcore >> 4) & 0x3FFF) << 16;   // leading byte offset: K-adjacent cores
  d |= (uint64_t)((rgroup >> 4) & 0x3FFF) << 32;  // stride byte offset: row-adjacent 8-row groups
  d |= (uint64_t)1 << 46;                         // descriptor version (fixed 0b001 at bits 46-48)
  return d;                                       // base offset 0, relative offsets, no swizzle
}
// kind::f16 instruction descriptor: D in FP32, A and B both FP16 (bf = 0) or both BF16 (bf = 1),
// both K-major, N >> 3 at bit 17, M >> 4 at bit 24
__host__ __device__ constexpr unsigned umma_idesc(int bf, int m, int n) {
  return (1u << 4) | ((unsigned)bf << 7) | ((unsigned)bf << 10) | ((unsigned)(n >> 3) << 17) |
         ((unsigned)(m >> 4) << 24);
}
__device__ __forceinline__ void umma(unsigned dtmem, uint64_t a, uint64_t b, unsigned idesc, unsigned accumulate) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(
          dtmem),
      "l"(a), "l"(b), "r"(idesc), "r"(accumulate)
      : "memory");
}
__device__ __forceinline__ void umma_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
               : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

#define DG_TMEM_R8(i) "=r"(r[i + 0]), "=r"(r[i + 1]), "=r"(r[i + 2]), "=r"(r[i + 3]), "=r"(r[i + 4]), "=r"(r[i + 5]), \
                      "=r"(r[i + 6]), "=r"(r[i + 7])
// 16 consecutive FP32 columns of this thread's TMEM lane
__device__ __forceinline__ void tmem_ld16(unsigned taddr, unsigned (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : DG_TMEM_R8(0), DG_TMEM_R8(8)
      : "r"(taddr)
      : "memory");
}
#undef DG_TMEM_R8
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

template <int BF>
__device__ __forceinline__ unsigned short to16(float x) {
  if constexpr (BF) {
    const __nv_bfloat16 h = __float2bfloat16_rn(x);
    return *reinterpret_cast<const unsigned short*>(&h);
  } else {
    const __half h = __float2half_rn(x);
    return *reinterpret_cast<const unsigned short*>(&h);
  }
}

__device__ __forceinline__ float pow2_scale(float mx) {  // 2^-ceil(log2 mx): brings mx into (1/2, 1]
  if (!(mx > 0.0f) || !isfinite(mx)) return 1.0f;
  int ex;
  frexpf(mx, &ex);  // mx = f 2^ex, f in [1/2, 1)
  return ldexpf(1.0f, -ex);
}

struct TcVolArgs {
  MeshDev M;
  const float* wvol;
  const float* in;
  float* out;
  const float* face_buf;
  const float* ubar;
  const float* ubar_scale;
  const uint4* tab;  // TA1 then TB2, 16-bit, in the operand layout (kTabBytes)
  float nu;
  double inv_gdt;
  unsigned* status;
  unsigned wait_polls;
};

// Pointwise products of the elements EL0 .. EL0 + NEL - 1 (NEL <= 5) at this thread's Gauss point q:
// their interpolated (scaled) velocity variation sits in TMEM columns 3 el + f.
template <int K, int BF, int EL0, int NEL>
__device__ __forceinline__ void tc_pointwise(const TcVolArgs& a, unsigned tmem_lane, int q, int e0, int cnt,
                                             const float* sTau, float wq, unsigned char* sm) {
  using Z = TcSz<K>;
  unsigned r[16];
  tmem_ld16(tmem_lane + 3 * EL0, r);
  const bool qv = q < Z::NQ;
  float ub[NEL][3];
#pragma unroll
  for (int j = 0; j < NEL; ++j) {
    const bool ok = qv && EL0 + j < cnt;
#pragma unroll
    for (int c = 0; c < 3; ++c) ub[j][c] = ok ? __ldg(a.ubar + ((size_t)(e0 + EL0 + j) * 3 + c) * Z::NQ + q) : 0.0f;
  }
  tmem_wait_ld();
#pragma unroll
  for (int j = 0; j < NEL; ++j) {
    const int el = EL0 + j;
    const bool ok = qv && el < cnt;
    const float tw = sTau[el] * wq;
    float u[3], b[3];
#pragma unroll
    for (int f = 0; f < 3; ++f) {
      u[f] = __uint_as_float(r[3 * j + f]);
      b[f] = tw * ub[j][f];
    }
    unsigned char* A2 = sm + kA2 + core_off(0, q, kKcA2, kRgA2);
#pragma unroll
    for (int sp = 0; sp < 6; ++sp) {
      const int p = sp < 3 ? sp : (sp == 5 ? 1 : 0), i = sp < 3 ? sp : (sp == 3 ? 1 : 2);
      const float v = ok ? u[p] * b[i] + b[p] * u[i] : 0.0f;
      *reinterpret_cast<unsigned short*>(A2 + core_off(6 * el + sp, 0, kKcA2, kRgA2)) = to16<BF>(v);
    }
  }
}

template <int K, int BF>
__global__ void __launch_bounds__(kTcThreads, 4) tc_vol_kernel(TcVolArgs a) {
  if (!wait_previous()) return;
  using Z = TcSz<K>;
  constexpr int NB = Z::NB, NBM = Z::NBM, NT = Z::NT, NQ = Z::NQ, N2 = Z::N2, LD = Z::LD;
  extern __shared__ __align__(1024) unsigned char sm[];
  __shared__ uint64_t bar;
  __shared__ unsigned tslot;
  __shared__ float sSig[kTcE], sTau[kTcE];
  float* sC = reinterpret_cast<float*>(sm + Z::SC);
  float* sT = reinterpret_cast<float*>(sm + Z::ST);
  float* sGeo = reinterpret_cast<float*>(sm + Z::GE);
  int* sFid = reinterpret_cast<int*>(sm + Z::FID);
  float* sG = reinterpret_cast<float*>(sm + kA2);  // corrected gradient, while the products' buffer is idle
  float* sO = sG;                                  // output rows, after the integration MMA
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, nt = blockDim.x, nw = nt >> 5;
  const int ne = a.M.ne, ntiles = (ne + kTcE - 1) / kTcE;

  if (tid == 0) mbar_init(&bar, 1);
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tslot)),
                 "r"(kTcCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  // the basis tables (16-bit operands), zeroed interpolation operand (its K padding stays zero)
  {
    uint4* s4 = reinterpret_cast<uint4*>(sm);
    for (int i = tid; i < (int)(kTabBytes / 16); i += nt) s4[kTA1 / 16 + i] = a.tab[i];
    for (int i = tid; i < (int)(kB1Bytes / 16); i += nt) s4[kB1 / 16 + i] = make_uint4(0, 0, 0, 0);
  }
  float* sS = reinterpret_cast<float*>(sm + Z::SS);
  float* sI = sS + NB;
  for (int t = tid; t < NB; t += nt) {
    sS[t] = mode_scale<float, K>.s[t];
    sI[t] = mode_scale<float, K>.inv[t];
  }
  fence_proxy_async_smem();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const unsigned tmem = tslot;
  const unsigned lane_base = (unsigned)(32 * (warp & 3)) << 16;
  const unsigned sbase = smem_u32(sm);
  const int q = 32 * (warp & 3) + lane;
  const float wq = q < NQ ? a.wvol[q] : 0.0f;
  unsigned phase = 0;
  bool nonfinite = false;

  for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    const int e0 = tile * kTcE;
    const int cnt = min(kTcE, ne - e0);
    if (tid == 0 && tile + (int)gridDim.x < ntiles) {
      // the next tile's contiguous inputs into L2 while this tile is computed
      const int n0 = (tile + gridDim.x) * kTcE, n1 = min(ne, n0 + kTcE);
      prefetch_l2(a.in + (size_t)n0 * 4 * NB, a.in + (size_t)n1 * 4 * NB);
      prefetch_l2(a.face_buf + face_record<N2>(face_slot(n0, 0), 0), a.face_buf + face_record<N2>(face_slot(n0, 0), 0) + 21 * N2 * kFaceGroup);
      prefetch_l2(a.ubar + (size_t)n0 * 3 * NQ, a.ubar + (size_t)n1 * 3 * NQ);
    }
    // 1. scaled coefficients, geometry and face records
    Z::fetch(a.in, e0, cnt, sC, tid, nt);
    Z::meta(a.M, a.inv_gdt, e0, cnt, sGeo, sFid, tid, nt);
    if (tid < kTcE) sTau[tid] = tid < cnt ? a.ubar_scale[e0 + tid] : 1.0f;
    Z::scale(sS, sC, tid, nt);
    __syncthreads();
    // the scale sigma of the element's velocity and its rows (e, f) of the interpolation's B operand
    for (int e = warp; e < kTcE; e += nw) {
      constexpr int NV = (3 * NB + 31) / 32;
      float v[NV], mx = 0.0f;
#pragma unroll
      for (int k = 0; k < NV; ++k) {
        const int m = lane + 32 * k;
        v[k] = m < 3 * NB ? sC[m * LD + e] : 0.0f;
        mx = fmaxf(mx, fabsf(v[k]));
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
      const float sg = pow2_scale(mx);
      if (lane == 0) sSig[e] = sg;
#pragma unroll
      for (int k = 0; k < NV; ++k) {
        const int m = lane + 32 * k, f = m / NB;
        if (m < 3 * NB)
          *reinterpret_cast<unsigned short*>(sm + kB1 + core_off(3 * e + f, m - f * NB, kKc, kRgB1)) = to16<BF>(sg * v[k]);
      }
    }
    fence_proxy_async_smem();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (tid == 0) {
      constexpr unsigned id1 = umma_idesc(BF, 128, kN1);
#pragma unroll
      for (int kk = 0; kk < kMP / 16; ++kk)
        umma(tmem, umma_smem_desc(sbase + kTA1 + kk * 2 * kKc, kKc, kRgTA1),
             umma_smem_desc(sbase + kB1 + kk * 2 * kKc, kKc, kRgB1), id1, kk > 0);
      umma_commit(&bar);
    }
    // 2. while the MMA runs: corrected gradients (into the idle products' buffer), viscous flux
    Z::gradient(sC, a.face_buf, sGeo, sFid, a.nu, sG, warp, nw, lane);
    __syncthreads();
    Z::viscous(sC, sG, sT, warp, nw, lane);
    // 3. the interpolated velocity variation: wait for the MMA
    bool ok = mbar_wait(&bar, phase & 1, a.wait_polls);
    ++phase;
    if (!__syncthreads_and(ok)) {
      if (tid == 0) {
        atomicOr(a.status, (unsigned)DG_STATUS_WAIT);
        mbar_wait(&bar, (phase - 1) & 1);  // the MMA in flight lands before the tensor memory is freed
      }
      break;
    }
    tc_fence_after();
    // 4. pointwise products into the integration's A operand (sG is no longer needed)
    if (warp < 4)
      tc_pointwise<K, BF, 0, 4>(a, tmem + lane_base, q, e0, cnt, sTau, wq, sm);
    else
      tc_pointwise<K, BF, 4, kTcE - 4>(a, tmem + lane_base, q, e0, cnt, sTau, wq, sm);
    fence_proxy_async_smem();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (tid == 0) {
      constexpr unsigned id2 = umma_idesc(BF, 128, kN2);
#pragma unroll
      for (int kk = 0; kk < kQP / 16; ++kk)
        umma(tmem + kTcD2, umma_smem_desc(sbase + kA2 + kk * 2 * kKcA2, kKcA2, kRgA2),
             umma_smem_desc(sbase + kTB2 + kk * 2 * kKc, kKc, kRgTB2), id2, kk > 0);
      umma_commit(&bar);
    }
    ok = mbar_wait(&bar, phase & 1, a.wait_polls);
    ++phase;
    if (!__syncthreads_and(ok)) {
      if (tid == 0) {
        atomicOr(a.status, (unsigned)DG_STATUS_WAIT);
        mbar_wait(&bar, (phase - 1) & 1);
      }
      break;
    }
    tc_fence_after();
    // 5. the products' coefficients, unscaled (D2 / (sigma tau)), taken off the viscous flux: sixteen
    // modes per group of four warps, the two lane quarters that hold rows in use
    if ((warp & 3) < (6 * kTcE + 31) / 32 && 16 * (warp >> 2) < NBM) {
      const int m0 = 16 * (warp >> 2), el = q / 6, sp = q - 6 * el;
      unsigned r[16];
      tmem_ld16(tmem + lane_base + kTcD2 + m0, r);
      tmem_wait_ld();
      if (el < cnt) {
        const float inv = 1.0f / (sSig[el] * sTau[el]);
        float* t = sT + (sp * NT + m0) * LD + el;
#pragma unroll
        for (int m = 0; m < 16; ++m)
          if (m0 + m < NBM) t[m * LD] -= __uint_as_float(r[m]) * inv;
      }
    }
    tc_fence_before();
    __syncthreads();
    // 6. modal derivatives of the fluxes and the face terms; output
    Z::divergence(sC, sT, a.face_buf, sGeo, sFid, sO, warp, nw, lane);
    __syncthreads();
    nonfinite |= Z::template store<true>(a.in, a.out, e0, cnt, sI, sO, sGeo, tid, nt);
    __syncthreads();  // the next tile rewrites the geometry and, after a barrier, the output rows
  }
  if (nonfinite && a.status) atomicOr(a.status, (unsigned)DG_STATUS_NONFINITE);
  tc_fence_before();
  __syncthreads();
  if (warp == 0)  // always released: a CTA must not exit holding tensor memory
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTcCols) : "memory");
}

// one warp per element: tau_e = 2^-ceil(log2 max |ub|) over the element's linearisation velocity
__global__ void ubar_scale_kernel(int ne, int n3q, const float* __restrict__ ubar, float* __restrict__ scale) {
  const int lane = threadIdx.x & 31;
  for (int e = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; e < ne; e += (gridDim.x * blockDim.x) >> 5) {
    float mx = 0.0f;
    for (int t = lane; t < n3q; t += 32) mx = fmaxf(mx, fabsf(ubar[(size_t)e * n3q + t]));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    if (lane == 0) scale[e] = pow2_scale(mx);
  }
}

template <int K, int BF>
int launch_tc(Handle* h, const TcVolArgs& a, cudaStream_t st) {
  const size_t smem = TcSz<K>::BYTES;
  DG_CUDA(h, cudaFuncSetAttribute(tc_vol_kernel<K, BF>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  const int ntiles = (h->ne + kTcE - 1) / kTcE;
  const int per_sm = (int)std::max<size_t>(1, std::min<size_t>(4, (227 * 1024) / (smem + 2048)));
  const int grid = std::min(ntiles, h->nsm * per_sm);
  launch(tc_vol_kernel<K, BF>, grid, kTcThreads, smem, st, a);
  DG_LAUNCH_CHECK(h);
  return DG_OK;
}

}  // namespace

// The 16-bit basis tables of the tensor-core volume pass (FP16 and BF16), from the FP64 table
// phi_hat_m(x_q) = s_m L_m(x_q): interpolation A operand L_m(x_q) [128 q][48 m] and integration B
// operand W_m L_m(x_q), W_m = prod (2 n_d + 1)/2 = s_m^2, [32 m][128 q] for the modes of degree
// <= k - 1, zero elsewhere. Once per handle; allocates, so it runs before any capture.
int tc_prepare_tables(Handle* h) {
  if (h->tc_tab[0] && h->tc_tab[1]) return DG_OK;
  const int nq = h->tab.nq, nb = h->tab.nb, nbm = nb_of(h->tab.k - 1);
  if (nq > kQP || nb > kMP || nbm > kN2) return fail(h, DG_ERR_ARG, "degree unsuited to the tensor-core volume pass");
  std::vector<double> B((size_t)nq * nb);
  std::vector<int> md((size_t)3 * nb);
  DG_CUDA(h, cudaMemcpy(B.data(), h->tab.Bvol, sizeof(double) * B.size(), cudaMemcpyDeviceToHost));
  DG_CUDA(h, cudaMemcpy(md.data(), h->tab.md3, sizeof(int) * md.size(), cudaMemcpyDeviceToHost));
  for (int bf = 0; bf < 2; ++bf) {
    std::vector<unsigned short> T(kTabBytes / 2, 0);
    auto put = [&](unsigned byte_off, double v) {
      unsigned short u;
      if (bf) {
        const __nv_bfloat16 x = __float2bfloat16_rn((float)v);
        u = *reinterpret_cast<const unsigned short*>(&x);
      } else {
        const __half x = __float2half_rn((float)v);
        u = *reinterpret_cast<const unsigned short*>(&x);
      }
      T[byte_off / 2] = u;
    };
    for (int m = 0; m < nb; ++m) {
      const double s = leg_scale(md[3 * m]) * leg_scale(md[3 * m + 1]) * leg_scale(md[3 * m + 2]);
      for (int qq = 0; qq < nq; ++qq) {
        const double v = B[(size_t)qq * nb + m];
        put(core_off(qq, m, kKc, kRgTA1), v / s);
        if (m < nbm) put(kTB2 - kTA1 + core_off(m, qq, kKc, kRgTB2), v * s);
      }
    }
    DG_CUDA(h, cudaMalloc(&h->tc_tab[bf], kTabBytes));
    DG_CUDA(h, cudaMemcpy(h->tc_tab[bf], T.data(), kTabBytes, cudaMemcpyHostToDevice));
  }
  return DG_OK;
}

// per-element scale of the FP32 linearisation velocity (after prepare_lin_fp32 refreshed it)
int tc_prepare_lin(Handle* h, cudaStream_t st) {
  if (!h->ubar_scale) DG_CUDA(h, cudaMalloc(&h->ubar_scale, sizeof(float) * (size_t)h->ne));
  const int n3q = 3 * h->tab.nq;
  const int grid = std::min(h->nsm * 8, (h->ne * 32 + 255) / 256);
  ubar_scale_kernel<<<grid, 256, 0, st>>>(h->ne, n3q, h->ubar_f, h->ubar_scale);
  DG_LAUNCH_CHECK(h);
  return DG_OK;
}

// Volume pass of the FP32 Jacobian action on the tensor cores; the face pass has run (its
// records are in face_buf_f). tc = 1: FP16 operands, tc = 2: BF16 operands.
int tc_volume_tangent(Handle* h, const float* in, float* out, int tc, cudaStream_t st) {
  if (!h->tc_tab[0] || !h->ubar_scale) return fail(h, DG_ERR_STATE, "tensor-core tables not prepared");
  const int bf = tc == 2 ? 1 : 0;
  TcVolArgs a;
  a.M = mesh_dev(h);
  a.wvol = h->tabf.wvol;
  a.in = in;
  a.out = out;
  a.face_buf = h->face_buf_f;
  a.ubar = h->ubar_f;
  a.ubar_scale = h->ubar_scale;
  a.tab = static_cast<const uint4*>(h->tc_tab[bf]);
  a.nu = (float)h->p.nu;
  a.inv_gdt = h->inv_gdt;
  a.status = h->status;
  a.wait_polls = h->dbg.wait_polls > 0 ? (unsigned)h->dbg.wait_polls : kBulkWaitLimit;
  switch (h->tab.k) {
    case 1: return bf ? launch_tc<1, 1>(h, a, st) : launch_tc<1, 0>(h, a, st);
    case 2: return bf ? launch_tc<2, 1>(h, a, st) : launch_tc<2, 0>(h, a, st);
    case 3: return bf ? launch_tc<3, 1>(h, a, st) : launch_tc<3, 0>(h, a, st);
    case 4: return bf ? launch_tc<4, 1>(h, a, st) : launch_tc<4, 0>(h, a, st);
  }
  return fail(h, DG_ERR_ARG, "unsupported degree");
}

}  // namespace dg
