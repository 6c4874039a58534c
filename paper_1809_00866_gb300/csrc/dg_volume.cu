// Volume pass of the matrix-free DG operator (Eq. (NSdiscrRes), Eqs. (jacTrilFnotNU), (jacTrilnu)):
// corrected gradients grad u - R^K(u), the viscous, pressure and continuity terms as exact modal
// derivatives (F^nu is linear, p and u are polynomials of degree k), the convective term u (x) u by
// sum-factorised interpolation to and projection from the Gauss points, the six face contributions
// and the mass shift. All of it equals the quadrature form up to rounding, because the Gauss rule
// with k+1 points integrates every polynomial product done exactly here.
//
// Bound: GB300's FP64 pipe for double (2 FMA per clock and SM), issue for float. So the kernel
// spends as few arithmetic instructions as the method needs and keeps every lane of them busy:
//  * plain Legendre coefficients and even/odd pencils with constant tables (dg_pencil.h);
//  * a test function of degree k meets the fluxes only through its derivative, of degree k - 1, so
//    gradients, viscous fluxes and projections of the products are formed for the modes of degree
//    <= k - 1 alone (20 of 35 at k = 4);
//  * the third interpolation step, the six products and the first projection step are one phase, a
//    pencil of Gauss points per thread, in registers;
//  * E elements per CTA: the items of a phase are (pencil, element) pairs sorted by pencil length,
//    so a warp runs one length and its 32 lanes are busy also where one element has few pencils.
// At 32^3 P4, one element per CTA with table look-ups -> now (events included): FP64 1345 -> 659 us (9223
// operations per element, 0.87 of the measured FP64 rate), FP32 213 -> 68 us.
#include <algorithm>

#include "dg_async.h"
#include "dg_launch.h"
#include "dg_opargs.h"
#include "dg_volume_phases.h"

namespace dg {
namespace {

template <int K, class R, int E>
struct VolSmem : VolPhases<K, R, E> {
  using Ph = VolPhases<K, R, E>;
  using Ph::GEO, Ph::LD, Ph::N1, Ph::NB, Ph::NN, Ph::NT;
  // X: planes of (K+1)^2 rows (PL apart, odd), the fields at the (q1, q2) points per x exponent a in
  // plane 3 a + f, then, in place, the products' projections in plane 6 a + sp: a thread of phase (3)
  // reads and writes one row of every plane
  static constexpr int PL = NN | 1;
  static constexpr int GROW = 3 * N1 * PL;  // rows of X that hold the gradient meanwhile
  static constexpr int mx(int a, int b) { return a > b ? a : b; }
  static constexpr int XROWS = mx(mx(6 * K * PL, GROW + 9 * NT), 4 * NB);
  static constexpr int C = 0;                  // [4][NB] scaled coefficients
  static constexpr int T = C + 4 * NB * LD;    // [6][NBM] symmetric flux pairs
  static constexpr int X = T + 6 * NT * LD;    // the sum factorisation's partial results, in place; then the output
  static constexpr int SC = X + XROWS * LD;    // [2][NB] mode scales and their inverses
  static constexpr int GE = SC + 2 * NB;       // [2 parities][E][GEO]
  static constexpr int REALS = GE + 2 * GEO * E;
  static constexpr int INTS = 12 * E;          // [2 parities][E][6] face numbers
  static constexpr size_t bytes() { return sizeof(R) * REALS + sizeof(int) * INTS; }
};

template <int K, int MODE, class R, int E>
__global__ void __launch_bounds__(256, sizeof(R) == 4 ? 3 : 2) vol_kernel(OpArgsT<R> a) {
  if (!wait_previous()) return;
  using L = VolSmem<K, R, E>;
  constexpr int N1 = L::N1, NN = L::NN, NQ = L::NQ, N2 = L::N2, NB = L::NB, NT = L::NT, PL = L::PL, LD = L::LD;
  constexpr bool kPoints = MODE != MODE_LINPART;
  extern __shared__ __align__(16) unsigned char smraw_[];
  R* sm = reinterpret_cast<R*>(smraw_);
  R* sC = sm + L::C;
  R* sT = sm + L::T;
  R* X = sm + L::X;
  int* sFid0 = reinterpret_cast<int*>(sm + L::REALS);
  const int tid = threadIdx.x, nt = blockDim.x, nw = nt >> 5, warp = tid >> 5, lane = tid & 31;
  R* sS = sm + L::SC;
  R* sI = sS + NB;
  for (int t = tid; t < NB; t += nt) {
    sS[t] = mode_scale<R, K>.s[t];
    sI[t] = mode_scale<R, K>.inv[t];
  }
  __syncthreads();
  bool nonfinite = false;
  const int ngrp = (a.M.ne + E - 1) / E;
  int par = 0;
  // the warp that starts the task list moves on with every group, so that the remainders of the
  // task lists fall on all four schedulers of the SM alike
  int vw = (warp + blockIdx.x) % nw;
  // the group's rows, copied while the previous group is stored, and its other inputs on their way to L2
  auto fetch = [&](int grp) {
    const int e0 = grp * E, cnt = min(E, a.M.ne - e0);
    L::fetch(a.in, e0, cnt, sC, tid, nt);
    if (tid == 0) {
      if constexpr (MODE == MODE_TAN)
        prefetch_l2(a.ubar + (size_t)e0 * 3 * NQ, a.ubar + (size_t)(e0 + cnt) * 3 * NQ);
      if constexpr (E == kFaceGroup) {
        const R* f = a.face_buf + face_record<N2>(face_slot(e0, 0), 0);
        prefetch_l2(f, f + 21 * N2 * kFaceGroup);
      }
    }
  };
  if ((int)blockIdx.x < ngrp) fetch(blockIdx.x);
  for (int grp = blockIdx.x; grp < ngrp; grp += gridDim.x, par ^= 1) {
    const int e0 = grp * E, cnt = min(E, a.M.ne - e0);
    R* sGeo = sm + L::GE + par * L::GEO * E;
    int* sFid = sFid0 + par * 6 * E;
    vw = vw + 1 == nw ? 0 : vw + 1;
    L::meta(a.M, a.inv_gdt, e0, cnt, sGeo, sFid, tid, nt);
    L::scale(sS, sC, tid, nt);
    __syncthreads();
    // (1) corrected gradient
    L::gradient(sC, a.face_buf, sGeo, sFid, a.nu, X + L::GROW * LD, vw, nw, lane);
    // interpolation along z and y: for every x exponent a the triangle of the (y, z) exponents at the
    // points, rows [(field, a)][q1 q2]
    if constexpr (kPoints)
      for_classes<K + 1>(vw, nw, lane, [](auto) { return 3 * E; }, [&](auto ac, int it) {
        constexpr int A = decltype(ac)::value, N = K + 1 - A;
        const int f = it / E, e = it - f * E;
        const R* ce = sC + f * NB * LD + e;
        R* x = X + (3 * A + f) * PL * LD + e;
        R c[tri(N)];
        static_for<tri(N)>([&](auto jc) {
          constexpr int J = decltype(jc)::value, GD = face_degree(J), z = J - tri(GD);
          c[J] = ce[mode_at(A, GD - z, z) * LD];
        });
        interp_triangle<K, N>(c, [&](int q1, int q2, R v) { x[(q1 * N1 + q2) * LD] = v; });
      });
    __syncthreads();
    // (2) viscous flux minus pressure
    L::viscous(sC, X + L::GROW * LD, sT, vw, nw, lane);
    if constexpr (kPoints) {
      __syncthreads();
      // (3) one pencil of points along x per thread: interpolation step 3, the products with the
      // linearisation velocity (or with itself), projection step 1; rows [(product, a)][q1 q2]
      for_classes<1>(vw, nw, lane, [](auto) { return NN * E; }, [&](auto, int it) {
        const int r = it / E, e = it - r * E;
        const bool on = e < cnt;
        R* x = X + r * LD + e;
        R u[3][N1], ub[3][N1];
#pragma unroll
        for (int f = 0; f < 3; ++f) {
          R c[N1];
#pragma unroll
          for (int n = 0; n < N1; ++n) c[n] = x[(3 * n + f) * PL * LD];
          interp_pencil<K, N1>(c, u[f]);
        }
        R* ug = a.ubar + (size_t)(e0 + (on ? e : 0)) * 3 * NQ + r;
        [[maybe_unused]] const R is = sGeo[8 * e];
#pragma unroll
        for (int f = 0; f < 3; ++f)
#pragma unroll
          for (int q = 0; q < N1; ++q) {
            if constexpr (MODE == MODE_TAN) {
              ub[f][q] = ug[f * NQ + q * NN];
            } else {
              ub[f][q] = is * u[f][q];
              if (MODE == MODE_RES_LIN && on) ug[f * NQ + q * NN] = ub[f][q];
            }
          }
#pragma unroll
        for (int sp = 0; sp < 6; ++sp) {
          const int p = sp < 3 ? sp : (sp == 5 ? 1 : 0), i = sp < 3 ? sp : (sp == 3 ? 1 : 2);
          R v[N1], o[K];
#pragma unroll
          for (int q = 0; q < N1; ++q) {
            v[q] = u[p][q] * ub[i][q];
            if (MODE == MODE_TAN && sp >= 3) v[q] += ub[p][q] * u[i][q];
          }
          // the linearised square 2 u_p ub_p takes its factor from the projection
          if (MODE == MODE_TAN && sp < 3) project_pencil<K, K, 0, true>(v, o);
          else project_pencil<K, K>(v, o);
#pragma unroll
          for (int n = 0; n < K; ++n) x[(6 * n + sp) * PL * LD] = o[n];
        }
      });
      __syncthreads();
      // (4) projection along y and z, taken off the viscous flux: in FP32 for every x exponent a the
      // points (q1 q2) onto the triangle of the (y, z) exponents in one thread's registers; in FP64,
      // where idle lanes cost pipe time (6 x 8 items are one and a half warps), in two steps
      if constexpr (sizeof(R) == 4) {
        for_classes<K>(vw, nw, lane, [](auto) { return 6 * E; }, [&](auto ac, int it) {
          constexpr int A = decltype(ac)::value, N = K - A;
          const int sp = it / E, e = it - sp * E;
          const R* x = X + (6 * A + sp) * PL * LD + e;
          R* t = sT + sp * NT * LD + e;
          R o[tri(N)];
          static_for<tri(N)>([&](auto jc) {
            constexpr int J = decltype(jc)::value, GD = face_degree(J), z = J - tri(GD);
            o[J] = t[mode_at(A, GD - z, z) * LD];
          });
          project_triangle<K, N, -1>([&](int q1, int q2) { return x[(q1 * N1 + q2) * LD]; }, o);
          static_for<tri(N)>([&](auto jc) {
            constexpr int J = decltype(jc)::value, GD = face_degree(J), z = J - tri(GD);
            t[mode_at(A, GD - z, z) * LD] = o[J];
          });
        });
      } else {
        for_classes<K>(vw, nw, lane, [](auto) { return 6 * N1 * E; }, [&](auto gc, int it) {
          constexpr int G = decltype(gc)::value, N = K - G;
          const int e = it % E, p = it / E, sp = p / N1, q2 = p - sp * N1;
          R* x = X + ((6 * G + sp) * PL + q2) * LD + e;
          R v[N1], o[N];
#pragma unroll
          for (int q = 0; q < N1; ++q) v[q] = x[q * N1 * LD];
          project_pencil<K, N>(v, o);
#pragma unroll
          for (int n = 0; n < N; ++n) x[n * N1 * LD] = o[n];
        });
        __syncthreads();
        for_classes<K>(vw, nw, lane, [](auto g) { return 6 * (decltype(g)::value + 1) * E; }, [&](auto gc, int it) {
          constexpr int G = decltype(gc)::value, N = K - G;
          const int e = it % E, p = it / E, sp = p / (G + 1), b = p - sp * (G + 1), ax = G - b;
          const R* x = X + ((6 * ax + sp) * PL + b * N1) * LD + e;
          R* t = sT + sp * NT * LD + e;
          R v[N1], o[N];
#pragma unroll
          for (int q = 0; q < N1; ++q) v[q] = x[q * LD];
#pragma unroll
          for (int n = 0; n < N; ++n) o[n] = t[mode_at(ax, b, n) * LD];
          project_pencil<K, N, -1>(v, o);
#pragma unroll
          for (int n = 0; n < N; ++n) t[mode_at(ax, b, n) * LD] = o[n];
        });
      }
    }
    __syncthreads();
    // (5) modal derivatives of the fluxes and the face terms; (6) output
    L::divergence(sC, sT, a.face_buf, sGeo, sFid, X, vw, nw, lane);
    __syncthreads();
    if (grp + (int)gridDim.x < ngrp) fetch(grp + gridDim.x);
    nonfinite |= L::template store<MODE == MODE_TAN>(a.in, a.out, e0, cnt, sI, X, sGeo, tid, nt);
    // the next group's first writes go to sC and the other parity's geometry, which (6) does not read
  }
  // scan of the outputs: a non-finite entry (from a non-finite input or an overflow) sets the
  // status bit, once per thread that wrote one
  if (nonfinite && a.status) atomicOr(a.status, (unsigned)DG_STATUS_NONFINITE);
}

template <int K, int MODE, class R, int E>
int launch_vol(Handle* h, const OpArgsT<R>& a, const OpTune& t, cudaStream_t st) {
  const size_t smem = VolSmem<K, R, E>::bytes();
  auto kern = vol_kernel<K, MODE, R, E>;
  DG_CUDA(h, cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  int per_sm = resident_ctas(reinterpret_cast<const void*>(kern), t.vol_threads, smem);
  if (per_sm < 1) per_sm = 1;
  if (t.vol_per_sm > 0 && per_sm > t.vol_per_sm) per_sm = t.vol_per_sm;
  const int grid = std::min((h->ne + E - 1) / E, h->nsm * per_sm);
  launch(kern, grid, t.vol_threads, smem, st, a);
  DG_LAUNCH_CHECK(h);
  return DG_OK;
}

template <int K, int MODE, class R>
int pass_m(Handle* h, const OpArgsT<R>& a, const OpTune& t, cudaStream_t st) {
  // Elements per CTA: the fewest of 2, 4, 8 that leave every SM at most one CTA (FP32, whose CTAs share
  // an SM better, four). Fewer shorten a phase of one CTA, more fill its lanes. Volume pass at P4, FP64, with
  // 2 / 4 / 8 per CTA (us, events included): 216 elements 28 / 31 / 41, 512 35 / 31 / 41, 1000 55 / 42 / 43,
  // 4096 177 / 139 / 112; FP32: 1000 12.0 / 12.4 / 13.5, 2197 18.9 / 14.2 / 14.7, 4096 24.5 / 20.6 / 16.4.
  const int per = sizeof(R) == 8 ? h->nsm : 4 * h->nsm;
  return h->ne <= 2 * per ? launch_vol<K, MODE, R, 2>(h, a, t, st)
         : h->ne <= 4 * per ? launch_vol<K, MODE, R, 4>(h, a, t, st)
                            : launch_vol<K, MODE, R, 8>(h, a, t, st);
}

template <int K, class R>
int pass_k(Handle* h, const OpArgsT<R>& a, int mode, const OpTune& t, cudaStream_t st) {
  if constexpr (sizeof(R) == 8) {
    switch (mode) {
      case MODE_RES: return pass_m<K, MODE_RES, R>(h, a, t, st);
      case MODE_RES_LIN: return pass_m<K, MODE_RES_LIN, R>(h, a, t, st);
      case MODE_LINPART: return launch_vol<K, MODE_LINPART, R, 8>(h, a, t, st);  // set-up only
    }
  }
  return pass_m<K, MODE_TAN, R>(h, a, t, st);
}

}  // namespace

template <class R>
int volume_pass(Handle* h, const OpArgsT<R>& a, int mode, const OpTune& t, cudaStream_t st) {
  switch (h->tab.k) {
    case 1: return pass_k<1, R>(h, a, mode, t, st);
    case 2: return pass_k<2, R>(h, a, mode, t, st);
    case 3: return pass_k<3, R>(h, a, mode, t, st);
    case 4: return pass_k<4, R>(h, a, mode, t, st);
  }
  return fail(h, DG_ERR_ARG, "unsupported degree");
}
template int volume_pass<double>(Handle*, const OpArgsT<double>&, int, const OpTune&, cudaStream_t);
template int volume_pass<float>(Handle*, const OpArgsT<float>&, int, const OpTune&, cudaStream_t);

}  // namespace dg
