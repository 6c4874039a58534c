// Face pass of the matrix-free DG operator (Eq. (NSdiscrRes), Eqs. (jacTrilFnotNU), (jacTrilnu)): per
// face s = (K, K') the traces of both sides as 2D modal coefficients on the face (collapse over the
// normal exponent, exact), point values only of the four fields that the nonlinear
// artificial-compressibility Riemann flux needs, the flux (exact star state by safeguarded Newton;
// in tangent mode its cached Jacobian) projected back onto the 2D modes, and the BR2 viscous face
// flux F^nu({grad u - eta r^s}) built exactly in 2D modal space, the lifting r^s([u]) being a
// diagonal scaling of the 2D jump coefficients.
//
// Output, once per face: face_buf[f][0..3] = 2D coefficients of the normal flux (momentum x, y, z,
// continuity), face_buf[f][4..6] = those of the velocity's jump, all of plain Legendre products. The
// volume pass scales them by the element's own A4/(2 s) and takes the sign of its side.
//
// Bound: GB300's FP64 pipe for double, issue and the cached Jacobian's bytes for float. F faces of
// one direction share a CTA: the items of a phase are (pencil, face) pairs sorted by pencil length,
// so every warp runs one compile-time path with full lanes (one warp per face left 7 to 17 of 32
// lanes idle in its phases), on plain Legendre coefficients with even/odd pencils (dg_pencil.h).
// The linearised flux takes 16 values and 18 multiply-adds per point instead of the 32 of the full
// 4 x 8 Jacobian, which also halves the cache that every Jacobian action streams.
//
// Conventions (also in the C ABI header): orthonormal modal basis phi_m = phi_hat_m(xi)/s,
// s = sqrt(|K|/8); the normal of a face points from K (lower index) to K'; [v] = v_K - v_K'; the
// lifting is defined by int r . tau = + int_s [v] {tau} . n so that grad u - R^K is the consistent
// gradient (Sec. 2.1).
#include <algorithm>

#include "dg_opargs.h"
#include "dg_pencil.h"
#include "dg_riemann.h"

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
  static constexpr int NB = nb_of(K), N1 = K + 1, NN = N1 * N1, N2 = N1 * (K + 2) / 2;
  static constexpr int LD = F + 1;             // faces of a row, odd: rows and faces both spread over the banks
  static constexpr int C = 0;                  // [2][4][NB] scaled coefficients of K and K'
  static constexpr int X = C + 8 * NB * LD;    // [8][NN] traces, then point values, fluxes, their projections, in place
  static constexpr int V = X + 8 * NN * LD;    // [3][3][N2] velocity: jump, sum (tangential part), mean normal derivative
  static constexpr int SC = V + 9 * N2 * LD;   // [NB] mode scales
  static constexpr int GEO = SC + NB;          // [2 parities][F][8] 1/s and 2/h_n of both sides, 2/h_t1, 2/h_t2
  static constexpr int REALS = GEO + 16 * F;
  static constexpr size_t bytes() { return sizeof(R) * REALS + sizeof(int) * 4 * F; }  // + [2][F][2] face, wall
};

template <int K, int MODE, class R, int F>
__global__ void __launch_bounds__(256, 2) face_kernel(OpArgsT<R> a) {
  using L = FaceSmem<K, R, F>;
  constexpr int NB = L::NB, N1 = L::N1, NN = L::NN, N2 = L::N2, LD = L::LD;
  extern __shared__ __align__(16) unsigned char smraw_[];
  R* sm = reinterpret_cast<R*>(smraw_);
  R* sC = sm + L::C;
  R* X = sm + L::X;
  R* sV = sm + L::V;
  R* sS = sm + L::SC;
  int* sId0 = reinterpret_cast<int*>(sm + L::REALS);
  const int tid = threadIdx.x, nt = blockDim.x, nw = nt >> 5, warp = tid >> 5, lane = tid & 31;
  for (int t = tid; t < NB; t += nt) sS[t] = R(mode_scale<K>.s[t]);
  __syncthreads();
  const R nu = R(a.nu);
  // groups of F faces: for F consecutive elements their + faces along x, y, z, one direction per
  // group (neighbouring CTAs share the elements); then the walls below the lowest row
  const int nblk = (a.M.ne + F - 1) / F, ngrp = 3 * nblk + (a.M.nbf + F - 1) / F;
  int par = 0;
  int vw = (warp + blockIdx.x) % nw;  // rotates with the groups, as in the volume pass
  for (int grp = blockIdx.x; grp < ngrp; grp += gridDim.x, par ^= 1) {
    R* sGeo = sm + L::GEO + par * 8 * F;
    int* sId = sId0 + par * 2 * F;
    vw = vw + 1 == nw ? 0 : vw + 1;
    const bool below = grp >= 3 * nblk;  // walls below: element on the + side, ghost on the - side
    const int blk = below ? grp - 3 * nblk : grp / 3, d = below ? 1 : grp - 3 * blk;
    const int t1 = d == 2 ? 0 : d + 1, t2 = d == 0 ? 2 : d - 1;
    const int f0 = blk * F, cnt = min(F, (below ? a.M.nbf : a.M.ne) - f0);
    // the elements of both sides; a wall face has one real element, read on both sides here
    auto sides = [&](int fl, int& el, int& er, int& wall) {
      const int i = f0 + (fl < cnt ? fl : 0);
      wall = 0;
      if (below) {
        el = er = a.M.bface[i];
        wall = 2;
      } else {
        el = i;
        er = a.M.nbr[(size_t)i * 6 + 2 * d + 1];
        if (er < 0) { er = i; wall = 1; }
      }
    };
    for (int t = tid; t < F * 8 * NB; t += nt) {
      const int fl = t / (8 * NB), r = t - fl * 8 * NB, sd = r >= 4 * NB;
      int el, er, wall;
      sides(fl, el, er, wall);
      const int m = r - sd * 4 * NB;
      sC[r * LD + fl] = fl < cnt ? a.in[(size_t)(sd ? er : el) * 4 * NB + m] * sS[m % NB] : R(0);
    }
    for (int fl = tid; fl < F; fl += nt) {
      int el, er, wall;
      sides(fl, el, er, wall);
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
    __syncthreads();
    // (1) traces: values of the four variables on both sides, [variable][b][c] with b, c the
    // exponents along t1, t2; of the velocity also the jump, the sum and the mean normal derivative.
    // At a wall the ghost side has the mirrored velocity, the real pressure and normal derivative,
    // and the tangential part is the real side's alone.
    for_classes<K + 1>(vw, nw, lane, [](auto g) { return 4 * (decltype(g)::value + 1) * F; }, [&](auto gc, int it) {
      constexpr int G = decltype(gc)::value, N = K + 1 - G;
      const int fl = it % F, p = it / F, v = p / (G + 1), c = p - v * (G + 1), b = G - c, j = tri(G) + c;
      int idx[N];
      pencil_modes(idx, d, G, b, c);
      const R* c0 = sC + v * NB * LD + fl;
      const R* c1 = c0 + 4 * NB * LD;
      const R* ge = sGeo + 8 * fl;
      const int wall = sId[2 * fl + 1];
      R v0 = R(0), v1 = R(0), d0 = R(0), d1 = R(0);
#pragma unroll
      for (int n = 0; n < N; ++n) {
        const R x0 = c0[idx[n] * LD], x1 = c1[idx[n] * LD];
        v0 = n ? v0 + x0 : x0;
        v1 = n ? (n % 2 ? v1 - x1 : v1 + x1) : x1;
        if (n && v < 3) {  // L_n'(1) = n (n+1) / 2, L_n'(-1) = (-1)^(n+1) n (n+1) / 2
          constexpr R kHalf = R(0.5);
          const R q = kHalf * R(n * (n + 1));
          d0 = n > 1 ? d0 + q * x0 : x0;
          d1 = n > 1 ? (n % 2 ? d1 + q * x1 : d1 - q * x1) : x1;
        }
      }
      v0 *= ge[0];
      v1 *= ge[1];
      R sum = v0 + v1;
      if (wall) {
        if (wall == 1) v1 = v < 3 ? -v0 : v0;
        else v0 = v < 3 ? -v1 : v1;
        sum = R(2) * (wall == 1 ? v0 : v1);
      }
      X[(v * NN + b * N1 + c) * LD + fl] = v0;
      X[((4 + v) * NN + b * N1 + c) * LD + fl] = v1;
      if (v < 3) {
        R n0 = d0 * (ge[0] * ge[2]), n1 = d1 * (ge[1] * ge[3]);
        if (wall == 1) n1 = n0;
        if (wall == 2) n0 = n1;
        R* o = sV + (v * N2 + j) * LD + fl;
        o[0] = v0 - v1;
        o[3 * N2 * LD] = sum;
        o[6 * N2 * LD] = R(0.5) * (n0 + n1);
      }
    });
    __syncthreads();
    if constexpr (MODE != MODE_LINPART) {
      // (2) the traces at the face points, along t2 then along t1, in place
      for_classes<K + 1>(vw, nw, lane, [](auto) { return 8 * F; }, [&](auto gc, int it) {
        constexpr int G = decltype(gc)::value, N = K + 1 - G;
        R* x = X + ((it / F) * NN + G * N1) * LD + it % F;
        R c[N], v[N1];
#pragma unroll
        for (int n = 0; n < N; ++n) c[n] = x[n * LD];
        interp_pencil<K, N>(c, v);
#pragma unroll
        for (int q = 0; q < N1; ++q) x[q * LD] = v[q];
      });
      __syncthreads();
      for_classes<1>(vw, nw, lane, [](auto) { return 8 * N1 * F; }, [&](auto, int it) {
        const int fl = it % F, p = it / F, s8 = p / N1, q2 = p - s8 * N1;
        R* x = X + (s8 * NN + q2) * LD + fl;
        R c[N1], v[N1];
#pragma unroll
        for (int n = 0; n < N1; ++n) c[n] = x[n * N1 * LD];
        interp_pencil<K, N1>(c, v);
#pragma unroll
        for (int q = 0; q < N1; ++q) x[q * N1 * LD] = v[q];
      });
      __syncthreads();
      // (3) the Riemann flux, or its linearisation, at the points, in the face's frame (n, t1, t2)
      for_classes<1>(vw, nw, lane, [](auto) { return NN * F; }, [&](auto, int it) {
        const int fl = it / NN, q = it - fl * NN;
        R* x = X + q * LD + fl;
        auto at = [&](int s, int v) { return x[(4 * s + v) * NN * LD]; };
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
        x[d * NN * LD] = Fn;
        x[t1 * NN * LD] = F1;
        x[t2 * NN * LD] = F2;
        x[3 * NN * LD] = Fp;
      });
      __syncthreads();
      // (4) their projection onto the 2D modes, along t1 then along t2, in place
      for_classes<1>(vw, nw, lane, [](auto) { return 4 * N1 * F; }, [&](auto, int it) {
        const int fl = it % F, p = it / F, i = p / N1, q2 = p - i * N1;
        R* x = X + (i * NN + q2) * LD + fl;
        R v[N1], o[N1];
#pragma unroll
        for (int q = 0; q < N1; ++q) v[q] = x[q * N1 * LD];
        project_pencil<K, N1>(v, o);
#pragma unroll
        for (int n = 0; n < N1; ++n) x[n * N1 * LD] = o[n];
      });
      __syncthreads();
      for_classes<K + 1>(vw, nw, lane, [](auto) { return 4 * F; }, [&](auto gc, int it) {
        constexpr int G = decltype(gc)::value, N = K + 1 - G;
        R* x = X + ((it / F) * NN + G * N1) * LD + it % F;
        R v[N1], o[N];
#pragma unroll
        for (int q = 0; q < N1; ++q) v[q] = x[q * LD];
        project_pencil<K, N>(v, o);
#pragma unroll
        for (int n = 0; n < N; ++n) x[n * LD] = o[n];
      });
      __syncthreads();
    }
    // (5) viscous face flux in 2D modal space, total flux and jump, one thread per 2D mode
    for_classes<1>(vw, nw, lane, [](auto) { return N2 * F; }, [&](auto, int it) {
      const int fl = it / N2, j = it - fl * N2;
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
      const R er = R(a.eta) * R(0.125) * (ge[2] + ge[3]) * R((K - g + 1) * (K - g + 1));
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
        R* o = a.face_buf + (size_t)sId[2 * fl] * 7 * N2 + j;
        auto conv = [&](int i) { return MODE == MODE_LINPART ? R(0) : X[(i * NN + b * N1 + c) * LD + fl]; };
        o[d * N2] = conv(d) - fd;
        o[t1 * N2] = conv(t1) - f1;
        o[t2 * N2] = conv(t2) - f2;
        R fp = conv(3);
        if (MODE == MODE_LINPART) fp = R(0);
        o[3 * N2] = fp;
#pragma unroll
        for (int v = 0; v < 3; ++v) o[(4 + v) * N2] = jump(v);
      }
    });
    // the next group's first writes go to sC and the other parity's geometry, which (5) does not read
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
  kern<<<std::min(groups, h->nsm * per_sm), threads, smem, st>>>(a);
  DG_LAUNCH_CHECK(h);
  return DG_OK;
}

template <int K, class R>
int pass_k(Handle* h, const OpArgsT<R>& a, int mode, const OpTune& t, cudaStream_t st) {
  const bool small = 3 * h->ne < 8 * h->nsm;
  if constexpr (sizeof(R) == 8) {
    switch (mode) {
      case MODE_RES: return small ? launch_face<K, MODE_RES, R, 2>(h, a, t, st) : launch_face<K, MODE_RES, R, 8>(h, a, t, st);
      case MODE_RES_LIN:
        return small ? launch_face<K, MODE_RES_LIN, R, 2>(h, a, t, st) : launch_face<K, MODE_RES_LIN, R, 8>(h, a, t, st);
      case MODE_LINPART:
        return small ? launch_face<K, MODE_LINPART, R, 2>(h, a, t, st) : launch_face<K, MODE_LINPART, R, 8>(h, a, t, st);
    }
  }
  return small ? launch_face<K, MODE_TAN, R, 2>(h, a, t, st) : launch_face<K, MODE_TAN, R, 8>(h, a, t, st);
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
