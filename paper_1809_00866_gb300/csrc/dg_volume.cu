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
#include <algorithm>

#include "dg_opargs.h"
#include "dg_pencil.h"

namespace dg {
namespace {

template <int K, class R, int E>
struct VolSmem {
  static constexpr int NB = nb_of(K), NBM = nb_of(K - 1), N1 = K + 1, NN = N1 * N1, NQ = NN * N1;
  static constexpr int N2 = N1 * (K + 2) / 2;
  static constexpr int LD = E + 1;  // elements of a row, odd: rows and elements both spread over the banks
  static constexpr int GROW = 3 * N1 * NN;  // rows of X that hold the gradient while T1 / T2 fill the first ones
  static constexpr int mx(int a, int b) { return a > b ? a : b; }
  static constexpr int XROWS = mx(mx(6 * K * NN, GROW + 9 * NBM), 4 * NB);
  static constexpr int C = 0;                  // [4][NB] scaled coefficients
  static constexpr int T = C + 4 * NB * LD;    // [6][NBM] symmetric flux pairs
  static constexpr int X = T + 6 * NBM * LD;   // the sum factorisation's partial results, in place; then the output
  static constexpr int SC = X + XROWS * LD;    // [2][NB] mode scales and their inverses
  static constexpr int GEO = SC + 2 * NB;      // [2 parities][E][8] 1/s, 2/h[3], A4/(2 s)[3], mass shift
  static constexpr int REALS = GEO + 16 * E;
  static constexpr size_t bytes() { return sizeof(R) * REALS + sizeof(int) * 12 * E; }  // + [2][E][6] face ids
};

template <int K, int MODE, class R, int E>
__global__ void __launch_bounds__(256, 2) vol_kernel(OpArgsT<R> a) {
  using L = VolSmem<K, R, E>;
  constexpr int NB = L::NB, NBM = L::NBM, N1 = L::N1, NN = L::NN, NQ = L::NQ, N2 = L::N2, LD = L::LD;
  constexpr bool kPoints = MODE != MODE_LINPART;
  extern __shared__ __align__(16) unsigned char smraw_[];
  R* sm = reinterpret_cast<R*>(smraw_);
  R* sC = sm + L::C;
  R* sT = sm + L::T;
  R* X = sm + L::X;
  R* sS = sm + L::SC;
  R* sI = sS + NB;
  int* sFid0 = reinterpret_cast<int*>(sm + L::REALS);
  const int tid = threadIdx.x, nt = blockDim.x, nw = nt >> 5, warp = tid >> 5, lane = tid & 31;
  for (int t = tid; t < NB; t += nt) {
    sS[t] = R(mode_scale<K>.s[t]);
    sI[t] = R(mode_scale<K>.inv[t]);
  }
  __syncthreads();
  bool nonfinite = false;
  const int ngrp = (a.M.ne + E - 1) / E;
  int par = 0;
  // the warp that starts the task list moves on with every group, so that the remainders of the
  // task lists fall on all four schedulers of the SM alike
  int vw = (warp + blockIdx.x) % nw;
  for (int grp = blockIdx.x; grp < ngrp; grp += gridDim.x, par ^= 1) {
    const int e0 = grp * E, cnt = min(E, a.M.ne - e0);
    R* sGeo = sm + L::GEO + par * 8 * E;
    int* sFid = sFid0 + par * 6 * E;
    vw = vw + 1 == nw ? 0 : vw + 1;
    // scaled coefficients (rows of a partly filled group are zero), geometry, face numbers
    for (int t = tid; t < E * 4 * NB; t += nt) {
      const int e = t / (4 * NB), r = t - e * 4 * NB;
      sC[r * LD + e] = e < cnt ? a.in[(size_t)e0 * 4 * NB + t] * sS[r % NB] : R(0);
    }
    for (int t = tid; t < 6 * E; t += nt) {
      const int e = t / 6, sl = t - 6 * e, d = sl >> 1, el = e0 + (e < cnt ? e : 0);
      int f = 3 * el + d;  // slot 2d+1: the element's own + face; 2d: its - neighbour's, or the wall below
      if (!(sl & 1)) {
        const int p = a.M.nbr[(size_t)el * 6 + sl];
        f = p >= 0 ? 3 * p + d : 3 * a.M.ne + a.M.bslot[el];
      }
      sFid[t] = f;
    }
    for (int e = tid; e < E; e += nt) {
      const R* g = geo_row<R>(a.M, e0 + (e < cnt ? e : 0));
      R* o = sGeo + 8 * e;
      o[0] = g[4];
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        o[1 + d] = g[5 + d];
        o[4 + d] = R(0.125) * g[(d + 1) % 3] * g[(d + 2) % 3] * g[4];
      }
      o[7] = R(a.inv_gdt * a.M.geo[(size_t)(e0 + (e < cnt ? e : 0)) * kGeo + 11]);
    }
    __syncthreads();
    // (1) nu times the corrected gradient, modes of degree <= K - 1: along axis d, with the
    // scaled jumps f of the two faces and alpha = A4 / (2 s),
    //   G_a = (2a+1) alpha/2 [4/s sum_{n = a+1, a+3, ..} c_n - (f_+ + (-1)^a f_-)]
    for_classes<K>(vw, nw, lane, [](auto g) { return 3 * (decltype(g)::value + 1) * E; }, [&](auto gc, int it) {
      constexpr int G = decltype(gc)::value, N = K + 1 - G;
      const int e = it % E, p = it / E, d = p / (G + 1), c = p - d * (G + 1), b = G - c, j = tri(G) + c;
      int idx[N];
      pencil_modes(idx, d, G, b, c);
      const R* ge = sGeo + 8 * e;
      const R is4 = R(4) * ge[0], beta = R(0.5) * R(a.nu) * ge[4 + d];
      const R* fp = a.face_buf + ((size_t)sFid[6 * e + 2 * d + 1] * 7 + 4) * N2 + j;
      const R* fm = a.face_buf + ((size_t)sFid[6 * e + 2 * d] * 7 + 4) * N2 + j;
      R bf[N - 1];
#pragma unroll
      for (int x = 0; x < N - 1; ++x) bf[x] = R(2 * x + 1) * beta;
#pragma unroll
      for (int av = 0; av < 3; ++av) {
        const R f1 = fp[av * N2], f0 = fm[av * N2];
        const R S = f1 + f0, D = f1 - f0;
        R sg[N + 1];
        sg[N - 1] = sg[N] = R(0);
#pragma unroll
        for (int x = N - 2; x >= 0; --x) {
          const R cn = sC[(av * NB + idx[x + 1]) * LD + e];
          sg[x] = x + 2 < N - 1 ? cn + sg[x + 2] : cn;
          X[(L::GROW + (av * 3 + d) * NBM + idx[x]) * LD + e] = bf[x] * (is4 * sg[x] - (x % 2 ? D : S));
        }
      }
    });
    // interpolation step 1, along z: rows [(field, a)][b][q2]
    if constexpr (kPoints)
      for_classes<K + 1>(vw, nw, lane, [](auto g) { return 3 * (decltype(g)::value + 1) * E; }, [&](auto gc, int it) {
        constexpr int G = decltype(gc)::value, N = K + 1 - G;
        const int e = it % E, p = it / E, f = p / (G + 1), b = p - f * (G + 1), ax = G - b;
        int idx[N];
        pencil_modes(idx, 2, G, ax, b);
        R c[N], v[N1];
#pragma unroll
        for (int x = 0; x < N; ++x) c[x] = sC[(f * NB + idx[x]) * LD + e];
        interp_pencil<K, N>(c, v);
#pragma unroll
        for (int q = 0; q < N1; ++q) X[((f * N1 + ax) * NN + b * N1 + q) * LD + e] = v[q];
      });
    __syncthreads();
    // (2) viscous flux minus pressure, nu (G_ip + G_pi - 2/3 delta tr G) - delta p, and
    // interpolation step 2, along y
    for_classes<1>(vw, nw, lane, [](auto) { return NBM * E; }, [&](auto, int it) {
      const int e = it % E, m = it / E;
      auto g = [&](int av, int b) { return X[(L::GROW + (av * 3 + b) * NBM + m) * LD + e]; };
      const R g00 = g(0, 0), g11 = g(1, 1), g22 = g(2, 2);
      const R tr = R(2.0 / 3.0) * (g00 + g11 + g22) + sC[(3 * NB + m) * LD + e];
      R* t = sT + m * LD + e;
      t[0 * NBM * LD] = R(2) * g00 - tr;
      t[1 * NBM * LD] = R(2) * g11 - tr;
      t[2 * NBM * LD] = R(2) * g22 - tr;
      t[3 * NBM * LD] = g(0, 1) + g(1, 0);
      t[4 * NBM * LD] = g(0, 2) + g(2, 0);
      t[5 * NBM * LD] = g(1, 2) + g(2, 1);
    });
    if constexpr (kPoints) {
      for_classes<K + 1>(vw, nw, lane, [](auto) { return 3 * N1 * E; }, [&](auto gc, int it) {
        constexpr int G = decltype(gc)::value, N = K + 1 - G;
        const int e = it % E, p = it / E, f = p / N1, q2 = p - f * N1;
        R* x = X + ((f * N1 + G) * NN + q2) * LD + e;
        R c[N], v[N1];
#pragma unroll
        for (int b = 0; b < N; ++b) c[b] = x[b * N1 * LD];
        interp_pencil<K, N>(c, v);
#pragma unroll
        for (int q = 0; q < N1; ++q) x[q * N1 * LD] = v[q];
      });
      __syncthreads();
      // (3) one pencil of points along x per thread: interpolation step 3, the products with the
      // linearisation velocity (or with itself), projection step 1; rows [(product, a)][q1 q2]
      for_classes<1>(vw, nw, lane, [](auto) { return NN * E; }, [&](auto, int it) {
        const int e = it / NN, r = it - e * NN;
        const bool on = e < cnt;
        R* x = X + r * LD + e;
        R u[3][N1], ub[3][N1];
#pragma unroll
        for (int f = 0; f < 3; ++f) {
          R c[N1];
#pragma unroll
          for (int n = 0; n < N1; ++n) c[n] = x[(f * N1 + n) * NN * LD];
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
          for (int n = 0; n < K; ++n) x[(sp * K + n) * NN * LD] = o[n];
        }
      });
      __syncthreads();
      // (4) projection step 2, along y, in place
      for_classes<K>(vw, nw, lane, [](auto) { return 6 * N1 * E; }, [&](auto gc, int it) {
        constexpr int G = decltype(gc)::value, N = K - G;
        const int e = it % E, p = it / E, sp = p / N1, q2 = p - sp * N1;
        R* x = X + ((sp * K + G) * NN + q2) * LD + e;
        R v[N1], o[N];
#pragma unroll
        for (int q = 0; q < N1; ++q) v[q] = x[q * N1 * LD];
        project_pencil<K, N>(v, o);
#pragma unroll
        for (int n = 0; n < N; ++n) x[n * N1 * LD] = o[n];
      });
      __syncthreads();
      // (5) projection step 3, along z, taken off the viscous flux
      for_classes<K>(vw, nw, lane, [](auto g) { return 6 * (decltype(g)::value + 1) * E; }, [&](auto gc, int it) {
        constexpr int G = decltype(gc)::value, N = K - G;
        const int e = it % E, p = it / E, sp = p / (G + 1), b = p - sp * (G + 1), ax = G - b;
        int idx[N];
        pencil_modes(idx, 2, G, ax, b);
        const R* x = X + ((sp * K + ax) * NN + b * N1) * LD + e;
        R* t = sT + sp * NBM * LD + e;
        R v[N1], o[N];
#pragma unroll
        for (int q = 0; q < N1; ++q) v[q] = x[q * LD];
#pragma unroll
        for (int n = 0; n < N; ++n) o[n] = t[idx[n] * LD];
        project_pencil<K, N, -1>(v, o);
#pragma unroll
        for (int n = 0; n < N; ++n) t[idx[n] * LD] = o[n];
      });
    }
    __syncthreads();
    // (6) modal derivatives of the fluxes (continuity: of -u) and the face terms, axis by axis:
    //   out_a += (2a+1) [2/h sum_{n = a-1, a-3, ..} T_n + alpha (F_+ - (-1)^a F_-)]
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      for_classes<K + 1>(vw, nw, lane, [](auto g) { return 4 * (decltype(g)::value + 1) * E; }, [&](auto gc, int it) {
        constexpr int G = decltype(gc)::value, N = K + 1 - G;
        const int e = it % E, p = it / E, i = p / (G + 1), c = p - i * (G + 1), b = G - c, j = tri(G) + c;
        int idx[N];
        pencil_modes(idx, d, G, b, c);
        const R* ge = sGeo + 8 * e;
        const R al = ge[4 + d], J = i == 3 ? -ge[1 + d] : ge[1 + d];
        const R fp = a.face_buf[((size_t)sFid[6 * e + 2 * d + 1] * 7 + i) * N2 + j];
        const R fm = a.face_buf[((size_t)sFid[6 * e + 2 * d] * 7 + i) * N2 + j];
        const R se = al * (fp - fm), so = al * (fp + fm);
        const R* t = (i == 3 ? sC + d * NB * LD : sT + (i == d ? d : i + d + 2) * NBM * LD) + e;
        R* o = X + i * NB * LD + e;
        R pi[N + 1];
        pi[0] = R(0);
#pragma unroll
        for (int x = 0; x < N; ++x) {
          if (x >= 1) {
            const R tn = t[idx[x - 1] * LD];
            pi[x] = x >= 3 ? tn + pi[x - 2] : tn;
          }
          const R s = x % 2 ? so : se;
          const R v = x ? J * pi[x] + s : s;
          o[idx[x] * LD] = d ? o[idx[x] * LD] + R(2 * x + 1) * v : R(2 * x + 1) * v;
        }
      });
      __syncthreads();
    }
    // (7) back to the orthonormal basis, mass shift, output
    for (int t = tid; t < cnt * 4 * NB; t += nt) {
      const int e = t / (4 * NB), r = t - e * 4 * NB;
      R v = X[r * LD + e] * sI[r % NB];
      if (MODE == MODE_TAN && r < 3 * NB) v += sGeo[8 * e + 7] * a.in[(size_t)e0 * 4 * NB + t];
      nonfinite |= !finite_bits(v);
      a.out[(size_t)e0 * 4 * NB + t] = v;
    }
    // the next group's first writes go to sC and the other parity's geometry, which (7) does not read
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
  kern<<<grid, t.vol_threads, smem, st>>>(a);
  DG_LAUNCH_CHECK(h);
  return DG_OK;
}

template <int K, class R>
int pass_k(Handle* h, const OpArgsT<R>& a, int mode, const OpTune& t, cudaStream_t st) {
  const bool small = h->ne < 8 * h->nsm;
  if constexpr (sizeof(R) == 8) {
    switch (mode) {
      case MODE_RES: return small ? launch_vol<K, MODE_RES, R, 2>(h, a, t, st) : launch_vol<K, MODE_RES, R, 8>(h, a, t, st);
      case MODE_RES_LIN:
        return small ? launch_vol<K, MODE_RES_LIN, R, 2>(h, a, t, st) : launch_vol<K, MODE_RES_LIN, R, 8>(h, a, t, st);
      case MODE_LINPART:
        return small ? launch_vol<K, MODE_LINPART, R, 2>(h, a, t, st) : launch_vol<K, MODE_LINPART, R, 8>(h, a, t, st);
    }
  }
  return small ? launch_vol<K, MODE_TAN, R, 2>(h, a, t, st) : launch_vol<K, MODE_TAN, R, 8>(h, a, t, st);
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
