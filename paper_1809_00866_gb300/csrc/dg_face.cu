// Face pass of the matrix-free DG operator (Eq. (NSdiscrRes), Eqs. (jacTrilFnotNU), (jacTrilnu)): per
// face s = (K, K') the traces of both sides as 2D modal coefficients on the face (collapse over the
// normal exponent, exact), point values only of the four fields that the nonlinear
// artificial-compressibility Riemann flux needs, the flux (exact star state, dg_riemann.h;
// in tangent mode its cached Jacobian) projected back onto the 2D modes, and the BR2 viscous face
// flux F^nu({grad u - eta r^s}) built exactly in 2D modal space, the lifting r^s([u]) being a
// diagonal scaling of the 2D jump coefficients.
//
// Output, once per face (face_record): 2D coefficients of the normal flux (momentum x, y, z,
// continuity) and of the velocity's jump, all of plain Legendre products. The volume pass scales them
// by the element's own A4/(2 s) and takes the sign of its side.
//
// Bound: GB300's FP64 pipe for double, issue and the shared-memory pipe for float. F faces of one
// direction share a CTA, so that every warp runs one compile-time path with full lanes (one warp per
// face left 7 to 17 of 32 lanes idle in its phases), on plain Legendre coefficients with even/odd
// pencils (dg_pencil.h). A thread takes one variable of one side of one face from its modal row to its
// point values in registers, and one flux component back; between them, one thread per point.
// The linearised flux takes 16 values and 18 multiply-adds per point instead of the 32 of the full
// 4 x 8 Jacobian, which also halves the cache that every Jacobian action streams.
// At 32^3 P4, one warp per face with table look-ups -> now (events included): FP64 tangent 1440 -> 665 us
// (9732 operations per element, 0.91 of the measured FP64 rate), FP32 tangent 208 -> 86 us, residual
// 5070 -> 1718 us.
//
// Conventions (also in the C ABI header): orthonormal modal basis phi_m = phi_hat_m(xi)/s,
// s = sqrt(|K|/8); the normal of a face points from K (lower index) to K'; [v] = v_K - v_K'; the
// lifting is defined by int r . tau = + int_s [v] {tau} . n so that grad u - R^K is the consistent
// gradient (Sec. 2.1).
#include <algorithm>

#include "dg_async.h"
#include "dg_launch.h"
#include "dg_opargs.h"
#include "dg_pencil.h"
#include "dg_riemann.h"
#include "dg_volume_phases.h"

namespace dg {
namespace {

// ---------------------------------------------------------------- face pass
__device__ __forceinline__ void load4g(const float* p, float* o) {
  const float4 v = __ldg(reinterpret_cast<const float4*>(p));
  o[0] = v.x; o[1] = v.y; o[2] = v.z; o[3] = v.w;
}
__device__ __forceinline__ void load4g(const double* p, double* o) {
  const double2 u = __ldg(reinterpret_cast<const double2*>(p)), v = __ldg(reinterpret_cast<const double2*>(p) + 1);
  o[0] = u.x; o[1] = u.y; o[2] = v.x; o[3] = v.y;
}

template <int K, class R, int F>
struct FaceSmem {
  static_assert(F % 4 == 0, "four faces, two sides and four variables share a warp");
  static constexpr int NB = nb_of(K), N1 = K + 1, NN = N1 * N1, N2 = N1 * (K + 2) / 2;
  // modal rows [side][face][4 NB]: a warp reads one mode of 4 faces x 4 variables x 2 sides; at
  // k = 4 (pitch 140 = 12 mod 32, variables 35 = 3 mod 32, sides 16 apart) from 32 different banks
  static constexpr int PC = K == 4 ? 4 * NB : 4 * NB + 2, SIDE = F * PC + 16;
  // points X[q][face / 4][side, variable][face % 4], 36 per four faces: the writes of a point by a
  // warp and the reads of a field by (face, point) pairs both hit 32 different banks
  static constexpr int PX = 36 * (F / 4);
  static constexpr int LD = F;                 // faces of a row of V and P
  static constexpr int C = 0;
  static constexpr int X = C + 2 * SIDE;
  static constexpr int V = X + NN * PX;        // [3][3][N2] velocity: jump, sum (tangential part), mean normal derivative
  static constexpr int P = V + 9 * N2 * LD;    // [4][N2] projected flux
  static constexpr int GEO = P + 4 * N2 * LD;  // [2 parities][F][8] 1/s and 2/h_n of both sides, 2/h_t1, 2/h_t2
  static constexpr int REALS = GEO + 16 * F;
  static constexpr int INTS = 4 * F;           // [2 parities][F][2] face of the flux Jacobian, wall
  static constexpr size_t bytes() { return sizeof(R) * REALS + sizeof(int) * INTS; }
};

__device__ __forceinline__ float flip_sign(float x, bool neg) {
  return __int_as_float(__float_as_int(x) ^ (neg ? 0x80000000 : 0));
}
__device__ __forceinline__ double flip_sign(double x, bool neg) {  // no FP64 instruction
  return __hiloint2double(__double2hiint(x) ^ (neg ? 0x80000000 : 0), __double2loint(x));
}

// Variable v of side `side` (0: element on the - side, its face at xi_D = 1) of one face: traces of the
// modal row c as 2D modes (b, x) along t1, t2, and their values at the face points to put(q1, q2, value)
// (POINTS). The lane with the other side is 16 away. Of the velocity, jump, sum and mean normal
// derivative go to vo. At a wall the ghost side has the mirrored velocity, the real pressure and normal
// derivative, and the tangential part is the real side's alone.
template <int K, int D, bool POINTS, class R, class Put>
__device__ __forceinline__ void face_traces(const R* c, int side, int v, int wall, R is, R jn, R* vo, int stride,
                                            Put put) {
  constexpr int NB = nb_of(K), N2 = (K + 1) * (K + 2) / 2;
  R t[N2], d[N2];
  static_for<NB>([&](auto mc) {
    constexpr int M = decltype(mc)::value, A = mode_exp(M, D), b = mode_exp(M, (D + 1) % 3),
                  x = mode_exp(M, (D + 2) % 3), J = tri(b + x) + x;
    // L_A(-1) = (-1)^A; L_A'(1) = A (A+1) / 2 and L_A'(-1) = -(-1)^A L_A'(1)
    R y = c[M] * mode_scale<R, K>.s[M];
    if constexpr (A % 2) y = flip_sign(y, side);
    t[J] = A ? t[J] + y : y;
    if constexpr (A >= 1) {
      constexpr double q = 0.5 * A * (A + 1);
      d[J] = A > 1 ? d[J] + R(q) * y : y;
    } else {
      d[J] = R(0);
    }
  });
  const R jd = flip_sign(R(0.5) * jn * is, side);
  const bool ghost = wall == 2 - side;  // wall 1: the + side, wall 2: the - side
#pragma unroll
  for (int j = 0; j < N2; ++j) {
    t[j] *= is;
    const R o = __shfl_xor_sync(0xffffffffu, t[j], 16);
    // the - side's lane forms the jump, the + side's the sum; at a wall the jump is twice the real
    // trace with the side's sign (the difference to the mirrored velocity), the sum twice the real one
    const R z = flip_sign(o, side == 0);
    const R w2 = (wall && ghost ? z : t[j]) + (wall && !ghost ? t[j] : z);
    if (ghost) t[j] = v < 3 ? -o : o;
    const bool has_n = j < tri(K);                        // modes of degree k have no normal derivative
    R n = has_n ? d[j] * jd : R(0);
    if (has_n) {
      const R on = __shfl_xor_sync(0xffffffffu, n, 16);
      n = wall ? R(2) * (ghost ? on : n) : n + on;
    }
    if (v < 3) {  // the - side's lane writes jump and normal derivative, the + side's the sum
      R* w = vo + j * stride;
      if (side == 0) {
        w[0] = w2;
        w[6 * N2 * stride] = n;
      } else {
        w[3 * N2 * stride] = w2;
      }
    }
  }
  if constexpr (POINTS) interp_triangle<K, K + 1>(t, put);
}

template <int K, int MODE, class R, int F>
__global__ void __launch_bounds__(256, sizeof(R) == 4 ? 3 : 2) face_kernel(OpArgsT<R> a) {
  if (!wait_previous()) return;
  using L = FaceSmem<K, R, F>;
  constexpr int NB = L::NB, N1 = L::N1, NN = L::NN, N2 = L::N2, LD = L::LD, PX = L::PX;
  extern __shared__ __align__(16) unsigned char smraw_[];
  R* sm = reinterpret_cast<R*>(smraw_);
  R* sC = sm + L::C;
  R* X = sm + L::X;
  R* sV = sm + L::V;
  R* sP = sm + L::P;
  int* sId0 = reinterpret_cast<int*>(sm + L::REALS);
  const int tid = threadIdx.x, nt = blockDim.x, nw = nt >> 5, warp = tid >> 5, lane = tid & 31;
  const R nu = a.nu, eta8 = a.eta8;
  auto cell = [](int fl, int s8) { return (fl >> 2) * 36 + s8 * 4 + (fl & 3); };
  // groups of F faces: for F consecutive elements their + faces along x, y, z, one direction per
  // group (neighbouring CTAs share the elements); then the walls below the lowest row
  const int nblk = (a.M.ne + F - 1) / F, ngrp = 3 * nblk + (a.M.nbf + F - 1) / F;
  struct Group {
    bool below;  // walls below: element on the + side, ghost on the - side
    int d, f0, cnt;
  };
  auto group = [&](int grp) {
    Group g;
    g.below = grp >= 3 * nblk;
    const int blk = g.below ? grp - 3 * nblk : grp / 3;
    g.d = g.below ? 1 : grp - 3 * blk;
    g.f0 = blk * F;
    g.cnt = min(F, (g.below ? a.M.nbf : a.M.ne) - g.f0);
    return g;
  };
  // the elements of both sides of face fl of a group; a wall face has one real element, read on both
  // sides here
  auto sides = [&](const Group& g, int fl, int& el, int& er, int& wall) {
    const int i = g.f0 + (fl < g.cnt ? fl : 0);
    wall = 0;
    if (g.below) {
      el = er = a.M.bface[i];
      wall = 2;
    } else {
      el = i;
      er = a.M.nbr[(size_t)i * 6 + 2 * g.d + 1];
      if (er < 0) { er = i; wall = 1; }
    }
  };
  // modal rows of both sides, one warp per (face, side), copied while the previous group is worked on
  // (the rows are free after its traces)
  auto fetch = [&](const Group& g) {
    for (int row = warp; row < 2 * F; row += nw) {
      const int fl = row >> 1, sd = row & 1;
      int el, er, wall;
      sides(g, fl, el, er, wall);
      const R* src = a.in + (size_t)(sd ? er : el) * 4 * NB;
      R* dst = sC + sd * L::SIDE + fl * L::PC;
      constexpr int W = 8 / sizeof(R);  // 8-byte copies: FP64 vectors are 8-byte aligned
#pragma unroll
      for (int k = 0; k < (4 * NB / W + 31) / 32; ++k) {
        const int m = (lane + 32 * k) * W;
        if (m < 4 * NB) async_value8(dst + m, src + m, fl < g.cnt);
      }
    }
    if constexpr (MODE == MODE_TAN) {  // and the flux Jacobian on its way to L2
      if (tid < g.cnt) {
        const size_t f = g.below ? 3 * (size_t)a.M.ne + g.f0 + tid : 3 * (size_t)(g.f0 + tid) + g.d;
        prefetch_l2(a.dFlux + f * 16 * NN, a.dFlux + (f + 1) * 16 * NN);
      }
    }
  };
  int par = 0;
  int vw = (warp + blockIdx.x) % nw;  // rotates with the groups, as in the volume pass
  if ((int)blockIdx.x < ngrp) fetch(group(blockIdx.x));
  for (int grp = blockIdx.x; grp < ngrp; grp += gridDim.x, par ^= 1) {
    R* sGeo = sm + L::GEO + par * 8 * F;
    int* sId = sId0 + par * 2 * F;
    vw = vw + 1 == nw ? 0 : vw + 1;
    const Group gr = group(grp);
    const bool below = gr.below;
    const int d = gr.d, f0 = gr.f0, cnt = gr.cnt;
    const int t1 = d == 2 ? 0 : d + 1, t2 = d == 0 ? 2 : d - 1;
    for (int fl = tid; fl < F; fl += nt) {
      int el, er, wall;
      sides(gr, fl, el, er, wall);
      const R* g0 = geo_row<R>(a.M, el);
      const R* g1 = geo_row<R>(a.M, er);
      R* o = sGeo + 8 * fl;
      o[0] = g0[4];
      o[1] = g1[4];
      o[2] = g0[5 + d];
      o[3] = g1[5 + d];
      o[4] = g0[5 + t1];
      o[5] = g0[5 + t2];
      sId[2 * fl] = below ? 3 * a.M.ne + f0 + fl : 3 * (f0 + fl) + d;
      sId[2 * fl + 1] = wall;
    }
    async_wait_all();
    __syncthreads();
    // (1) traces and their values at the face points: lane = (face % 4, variable, side)
    for_classes<1>(vw, nw, lane, [](auto) { return 8 * F; }, [&](auto, int it) {
      const int v = (it >> 2) & 3, side = (it >> 4) & 1, fl = (it >> 5) * 4 + (it & 3);
      const R* c = sC + side * L::SIDE + fl * L::PC + v * NB;
      R* vo = sV + v * N2 * LD + fl;
      R* x = X + cell(fl, 4 * side + v);
      auto put = [&](int q1, int q2, R val) { x[(q1 * N1 + q2) * PX] = val; };
      const int wall = sId[2 * fl + 1];
      const R is = sGeo[8 * fl + side], jn = sGeo[8 * fl + 2 + side];
      constexpr bool kPoints = MODE != MODE_LINPART;
      if (d == 0) face_traces<K, 0, kPoints>(c, side, v, wall, is, jn, vo, LD, put);
      else if (d == 1) face_traces<K, 1, kPoints>(c, side, v, wall, is, jn, vo, LD, put);
      else face_traces<K, 2, kPoints>(c, side, v, wall, is, jn, vo, LD, put);
    });
    __syncthreads();
    if (grp + (int)gridDim.x < ngrp) fetch(group(grp + gridDim.x));
    if constexpr (MODE != MODE_LINPART) {
      // (2) the Riemann flux, or its linearisation, at the points, in the face's frame (n, t1, t2)
      for_classes<1>(vw, nw, lane, [](auto) { return NN * F; }, [&](auto, int it) {
        const int q = it / F, fl = it - q * F;
        R* x = X + q * PX + cell(fl, 0);
        auto at = [&](int s, int v) { return x[(4 * s + v) * 4]; };
        const R ul = at(0, d), ur = at(1, d), pl = at(0, 3), pr = at(1, 3);
        const R l1 = at(0, t1), l2 = at(0, t2), r1 = at(1, t1), r2 = at(1, t2);
        R Fn, F1, F2, Fp;
        if constexpr (MODE == MODE_TAN) {
          R J[16] = {};
          if (fl < cnt) {
            const R* Jg = a.dFlux + ((size_t)sId[2 * fl] * 4 * NN + q) * 4;
#pragma unroll
            for (int i = 0; i < 4; ++i) load4g(Jg + i * NN * 4, J + 4 * i);
          }
          Fp = J[0] * ul + J[1] * pl + J[2] * ur + J[3] * pr;
          Fn = J[4] * ul + J[5] * pl + J[6] * ur + J[7] * pr;
          F1 = J[8] * Fp + J[12] * ul + J[13] * ur + J[10] * l1 + J[11] * r1;
          F2 = J[9] * Fp + J[14] * ul + J[15] * ur + J[10] * l2 + J[11] * r2;
        } else {  // residual modes run in FP64 only
          double Fr[4], J[16];
          ac_riemann(ul, l1, l2, pl, ur, r1, r2, pr, a.c, Fr, MODE == MODE_RES_LIN ? J : nullptr,
                     fl < cnt ? a.status : nullptr, a.riemann_its);
          Fn = Fr[0]; F1 = Fr[1]; F2 = Fr[2]; Fp = Fr[3];
          if (MODE == MODE_RES_LIN && fl < cnt) {
            R* Jg = a.dFlux + ((size_t)sId[2 * fl] * 4 * NN + q) * 4;
#pragma unroll
            for (int i = 0; i < 16; ++i) Jg[(i >> 2) * NN * 4 + (i & 3)] = J[i];
          }
        }
        x[d * 4] = Fn;
        x[t1 * 4] = F1;
        x[t2 * 4] = F2;
        x[3 * 4] = Fp;
      });
      __syncthreads();
      // (3) their projection onto the 2D modes: lane = (face % 4, component, ..)
      for_classes<1>(vw, nw, lane, [](auto) { return 4 * F; }, [&](auto, int it) {
        const int i = (it >> 2) & 3, fl = (it >> 4) * 4 + (it & 3);
        const R* x = X + cell(fl, i);
        R o[N2];
        project_triangle<K, N1>([&](int q1, int q2) { return x[(q1 * N1 + q2) * PX]; }, o);
#pragma unroll
        for (int j = 0; j < N2; ++j) sP[(i * N2 + j) * LD + fl] = o[j];
      });
      __syncthreads();
    }
    // (4) viscous face flux in 2D modal space, total flux and jump, one thread per 2D mode
    for_classes<1>(vw, nw, lane, [](auto) { return N2 * F; }, [&](auto, int it) {
      const int j = it / F, fl = it - j * F;
      int g = 0;
#pragma unroll
      for (int x = 1; x <= K; ++x) g += j >= tri(x);
      const int c = j - tri(g), b = g - c;
      const R* ge = sGeo + 8 * fl;
      const R* vj = sV + fl;
      auto jump = [&](int v) { return vj[(v * N2 + j) * LD]; };
      // {grad u}_n - eta {r^s}: the lifting of a jump mode of total degree g is
      // (k - g + 1)^2 / 4 (1/h_K + 1/h_K') [u], also at a wall ((k - g + 1)^2 / h_K times half the
      // difference to the mirrored ghost)
      const R er = eta8 * (ge[2] + ge[3]) * R((K - g + 1) * (K - g + 1));
      auto gn = [&](int v) { return vj[((6 + v) * N2 + j) * LD] - er * jump(v); };
      // d/dt of the mean trace: (2a+1) 2/h_t / 2 times the sum of the coefficients at a+1, a+3
      auto dt = [&](int v, int dir) {
        const R* s = vj + (3 + v) * N2 * LD;
        R acc = R(0);
#pragma unroll
        for (int n = 1; n <= K; n += 2)
          if (g + n <= K) acc += s[(tri(g + n) + c + (dir ? n : 0)) * LD];
        return acc * (R(0.5) * (dir ? ge[5] : ge[4]) * R(2 * (dir ? c : b) + 1));
      };
      const R gdd = gn(d), g11 = dt(t1, 0), g22 = dt(t2, 1);
      const R fd = nu * (R(2) * gdd - R(2.0 / 3.0) * (gdd + g11 + g22));
      const R f1 = nu * (gn(t1) + dt(d, 0)), f2 = nu * (gn(t2) + dt(d, 1));
      if (fl < cnt) {
        constexpr int C = N2 * kFaceGroup;  // components of a record
        R* o = a.face_buf + face_record<N2>(below ? wall_slot(a.M.ne, f0 + fl) : face_slot(f0 + fl, d), 0) + j * kFaceGroup;
        auto conv = [&](int i) { return MODE == MODE_LINPART ? R(0) : sP[(i * N2 + j) * LD + fl]; };
        o[d * C] = conv(d) - fd;
        o[t1 * C] = conv(t1) - f1;
        o[t2 * C] = conv(t2) - f2;
        o[3 * C] = conv(3);
#pragma unroll
        for (int v = 0; v < 3; ++v) o[(4 + v) * C] = jump(v);
      }
    });
    // the next group writes the other parity's geometry, and V and P only after a barrier
  }
}

template <int K, int MODE, class R, int F>
int launch_face(Handle* h, const OpArgsT<R>& a, const OpTune& t, cudaStream_t st) {
  const size_t smem = FaceSmem<K, R, F>::bytes();
  auto kern = face_kernel<K, MODE, R, F>;
  DG_CUDA(h, cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  const int threads = 32 * t.face_warps;
  int per_sm = resident_ctas(reinterpret_cast<const void*>(kern), threads, smem);
  if (per_sm < 1) per_sm = 1;
  if (t.face_per_sm > 0 && per_sm > t.face_per_sm) per_sm = t.face_per_sm;
  const int groups = 3 * ((h->ne + F - 1) / F) + (h->nbf + F - 1) / F;
  launch(kern, std::min(groups, h->nsm * per_sm), threads, smem, st, a);
  DG_LAUNCH_CHECK(h);
  return DG_OK;
}

template <int K, class R>
int pass_k(Handle* h, const OpArgsT<R>& a, int mode, const OpTune& t, cudaStream_t st) {
  // Faces per CTA: 4 while that gives an SM at most three groups of them (FP32: six), else 8. Face pass at
  // P4, FP64, with 4 / 8 (us, events included): 216 elements 22.8 / 24.6, 512 24.9 / 26.9, 1000 43.3 / 33.2;
  // FP32: 216 8.8 / 10.3, 1000 10.0 / 10.9, 1728 13.1 / 12.6.
  const bool small = 3 * h->ne <= (sizeof(R) == 8 ? 12 : 24) * h->nsm;
  if constexpr (sizeof(R) == 8) {
    switch (mode) {
      case MODE_RES: return small ? launch_face<K, MODE_RES, R, 4>(h, a, t, st) : launch_face<K, MODE_RES, R, 8>(h, a, t, st);
      case MODE_RES_LIN:
        return small ? launch_face<K, MODE_RES_LIN, R, 4>(h, a, t, st) : launch_face<K, MODE_RES_LIN, R, 8>(h, a, t, st);
      case MODE_LINPART:
        return small ? launch_face<K, MODE_LINPART, R, 4>(h, a, t, st) : launch_face<K, MODE_LINPART, R, 8>(h, a, t, st);
    }
  }
  return small ? launch_face<K, MODE_TAN, R, 4>(h, a, t, st) : launch_face<K, MODE_TAN, R, 8>(h, a, t, st);
}

}  // namespace

template <class R>
int face_pass(Handle* h, const OpArgsT<R>& a, int mode, const OpTune& t, cudaStream_t st) {
  switch (h->tab.k) {
    case 1: return pass_k<1, R>(h, a, mode, t, st);
    case 2: return pass_k<2, R>(h, a, mode, t, st);
    case 3: return pass_k<3, R>(h, a, mode, t, st);
    case 4: return pass_k<4, R>(h, a, mode, t, st);
  }
  return fail(h, DG_ERR_ARG, "unsupported degree");
}
template int face_pass<double>(Handle*, const OpArgsT<double>&, int, const OpTune&, cudaStream_t);
template int face_pass<float>(Handle*, const OpArgsT<float>&, int, const OpTune&, cudaStream_t);

}  // namespace dg
