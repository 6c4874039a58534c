// Phases of the volume pass that its two forms share (dg_volume.cu: sum factorisation on the CUDA
// cores; dg_tc_volume.cu: quadrature contractions on the tensor cores). A CTA works on E elements; rows
// of its shared arrays hold one value of all of them. Items are (something, element) pairs with the
// element fastest, also in the copies from and to memory, and the row counts that items stride over
// are odd: with E = 8 a warp's four groups of eight then fall on 32 different banks in every phase.
// (Rows of nine, dealt to the lanes mode by mode in the copies, cost 41 % of the shared-memory
// wavefronts in conflicts.) Each function is one phase without the barriers around it.
#pragma once

#include "dg_async.h"
#include "dg_pencil.h"

namespace dg {

template <int K, class R, int E>
struct VolPhases {
  static constexpr int NB = nb_of(K), NBM = nb_of(K - 1), N1 = K + 1, NN = N1 * N1, NQ = NN * N1;
  static constexpr int N2 = N1 * (K + 2) / 2, LD = E;
  static constexpr int NT = NBM | 1;               // rows of a gradient component or flux pair
  static constexpr int GEO = 8;                    // reals per element: 1/s, 2/h[3], A4/(2 s)[3], mass shift

  // asynchronous copy of the elements' rows (zero past the last element), and, once it has landed
  // (async_wait_all inside), their scaling by the same threads; sS: the mode scales
  static __device__ __forceinline__ void fetch(const R* in, int e0, int cnt, R* sC, int tid, int nt) {
    for (int t = tid; t < 4 * NB * E; t += nt) {
      const int m = t / E, e = t - m * E;
      async_value(sC + t, in + (size_t)(e0 + (e < cnt ? e : 0)) * 4 * NB + m, e < cnt);
    }
  }
  static __device__ __forceinline__ void scale(const R* sS, R* sC, int tid, int nt) {
    async_wait_all();
    for (int t = tid; t < 4 * NB * E; t += nt) sC[t] *= sS[t / E % NB];
  }

  // face records of the slots -x, +x, -y, ... (face_slot), geometry
  static __device__ __forceinline__ void meta(const MeshDev& M, double inv_gdt, int e0, int cnt, R* sGeo, int* sFid,
                                              int tid, int nt) {
    for (int t = tid; t < 6 * E; t += nt) {
      const int e = t / 6, sl = t - 6 * e, d = sl >> 1, el = e0 + (e < cnt ? e : 0);
      int f = face_slot(el, d);  // slot 2d+1: the element's own + face; 2d: its - neighbour's, or the wall below
      if (!(sl & 1)) {
        const int p = M.nbr[(size_t)el * 6 + sl];
        f = p >= 0 ? face_slot(p, d) : wall_slot(M.ne, M.bslot[el]);
      }
      sFid[t] = f;
    }
    for (int e = nt - 1 - tid; e < E; e += nt) {
      const int el = e0 + (e < cnt ? e : 0);
      const R* g = geo_row<R>(M, el);
      R* o = sGeo + GEO * e;
      o[0] = g[4];
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        o[1 + d] = g[5 + d];
        o[4 + d] = R(0.125) * g[(d + 1) % 3] * g[(d + 2) % 3] * g[4];
      }
      o[7] = R(inv_gdt * M.geo[(size_t)el * kGeo + 11]);
    }
  }

  // nu times the corrected gradient, modes of degree <= K - 1, rows (3 av + d) NT + mode of G:
  // along axis d, with the scaled jumps f of the two faces and alpha = A4 / (2 s),
  //   G_a = (2a+1) alpha/2 [4/s sum_{n = a+1, a+3, ..} c_n - (f_+ + (-1)^a f_-)]
  // One thread per (velocity component, element) and axis, every index fixed at compile time.
  static __device__ __forceinline__ void gradient(const R* sC, const R* face_buf, const R* sGeo, const int* sFid, R nu,
                                                  R* G, int vw, int nw, int lane) {
    for_classes<3>(vw, nw, lane, [](auto) { return 3 * E; }, [&](auto dc, int it) {
      constexpr int D = decltype(dc)::value;
      const int av = it / E, e = it - av * E;
      const R* ge = sGeo + GEO * e;
      const R is4 = R(4) * ge[0], beta = R(0.5) * nu * ge[4 + D];
      const R* fp = face_buf + face_record<N2>(sFid[6 * e + 2 * D + 1], 4 + av);
      const R* fm = face_buf + face_record<N2>(sFid[6 * e + 2 * D], 4 + av);
      const R* ce = sC + av * NB * LD + e;
      R* Ge = G + (av * 3 + D) * NT * LD + e;
      R bf[K], f1[tri(K)], f0[tri(K)], cn[NB];
#pragma unroll
      for (int x = 0; x < K; ++x) bf[x] = R(2 * x + 1) * beta;
#pragma unroll
      for (int j = 0; j < tri(K); ++j) {
        f1[j] = fp[j * kFaceGroup];
        f0[j] = fm[j * kFaceGroup];
      }
      // all loads before the first store, which the compiler would not move them across
      static_for<NB>([&](auto mc) {
        constexpr int M = decltype(mc)::value;
        if constexpr (mode_exp(M, D) >= 1) cn[M] = ce[M * LD];
      });
      static_for<tri(K)>([&](auto jc) {
        constexpr int J = decltype(jc)::value, GD = face_degree(J), c = J - tri(GD), b = GD - c, N = K + 1 - GD;
        const R S = f1[J] + f0[J], Df = f1[J] - f0[J];
        R sg[N + 1];
        sg[N - 1] = sg[N] = R(0);
        static_for<N - 1>([&](auto xc) {
          constexpr int X = N - 2 - decltype(xc)::value;
          constexpr int M = mode_along(D, X + 1, b, c);
          sg[X] = X + 2 < N - 1 ? cn[M] + sg[X + 2] : cn[M];
          Ge[mode_along(D, X, b, c) * LD] = bf[X] * (is4 * sg[X] - (X % 2 ? Df : S));
        });
      });
    });
  }

  // viscous flux minus pressure, nu (G_ip + G_pi - 2/3 delta tr G) - delta p: six symmetric pairs
  static __device__ __forceinline__ void viscous(const R* sC, const R* G, R* T, int vw, int nw, int lane) {
    for_classes<1>(vw, nw, lane, [](auto) { return NBM * E; }, [&](auto, int it) {
      const int e = it % E, m = it / E, o = m * LD + e;
      auto g = [&](int av, int b) { return G[(av * 3 + b) * NT * LD + o]; };
      const R g00 = g(0, 0), g11 = g(1, 1), g22 = g(2, 2);
      const R g01 = g(0, 1) + g(1, 0), g02 = g(0, 2) + g(2, 0), g12 = g(1, 2) + g(2, 1);
      const R tr = R(2.0 / 3.0) * (g00 + g11 + g22) + sC[3 * NB * LD + o];
      R* t = T + o;
      t[0 * NT * LD] = R(2) * g00 - tr;
      t[1 * NT * LD] = R(2) * g11 - tr;
      t[2 * NT * LD] = R(2) * g22 - tr;
      t[3 * NT * LD] = g01;
      t[4 * NT * LD] = g02;
      t[5 * NT * LD] = g12;
    });
  }

  // modal derivatives of the fluxes (continuity: of -u) and the face terms, rows i NB + mode of O:
  //   out_m = sum_d (2a+1) [2/h sum_{n = a-1, a-3, ..} T_n + alpha (F_+ - (-1)^a F_-)],  a = m_d
  // One thread per (equation, element) and part of the modes: z exponent 0, 1, or above. The split
  // by z exponents lets no part form another's x and y terms.
  static __device__ __forceinline__ void divergence(const R* sC, const R* T, const R* face_buf, const R* sGeo,
                                                    const int* sFid, R* O, int vw, int nw, int lane) {
    for_classes<(K > 1 ? 3 : 2)>(vw, nw, lane, [](auto) { return 4 * E; }, [&](auto pc, int it) {
      constexpr int PART = decltype(pc)::value;
      constexpr auto in_part = [](int m) { return PART < 2 ? mode_exp(m, 2) == PART : mode_exp(m, 2) >= 2; };
      const int i = it / E, e = it - i * E;
      const R* ge = sGeo + GEO * e;
      R fp[3][N2], fm[3][N2], out[NB];
      static_for<3>([&](auto dc) {
        constexpr int D = decltype(dc)::value;
        const R* gp = face_buf + face_record<N2>(sFid[6 * e + 2 * D + 1], i);
        const R* gm = face_buf + face_record<N2>(sFid[6 * e + 2 * D], i);
        static_for<N2>([&](auto jc) {
          constexpr int J = decltype(jc)::value, GD = face_degree(J), c = J - tri(GD), b = GD - c;
          // some mode along this pencil is in the part: b or c is the z exponent for D = 1 or 0
          constexpr bool need = D == 2 ? (PART < 2 ? GD + PART <= K : GD + 2 <= K)
                                       : (PART < 2 ? (D == 1 ? b : c) == PART : (D == 1 ? b : c) >= 2);
          if constexpr (need) {
            fp[D][J] = gp[J * kFaceGroup];
            fm[D][J] = gm[J * kFaceGroup];
          }
        });
      });
      static_for<NB>([&](auto mc) {
        constexpr int M = decltype(mc)::value;
        if constexpr (in_part(M)) {
          R acc = R(0);
          static_for<3>([&](auto dc) {
            constexpr int D = decltype(dc)::value, A = mode_exp(M, D), b = mode_exp(M, (D + 1) % 3),
                          c = mode_exp(M, (D + 2) % 3), J = tri(b + c) + c;
            const R* t = (i == 3 ? sC + D * NB * LD : T + (i == D ? D : i + D + 2) * NT * LD) + e;
            const R h = i == 3 ? -ge[1 + D] : ge[1 + D];
            R v = ge[4 + D] * (A % 2 ? fp[D][J] + fm[D][J] : fp[D][J] - fm[D][J]);
            if constexpr (A >= 1) {
              R pi = t[mode_along(D, A >= 1 ? A - 1 : 0, b, c) * LD];
              if constexpr (A >= 3) pi += t[mode_along(D, A >= 3 ? A - 3 : 0, b, c) * LD];
              v += h * pi;
            }
            acc = D ? acc + R(2 * A + 1) * v : R(2 * A + 1) * v;
          });
          out[M] = acc;
        }
      });
      R* o = O + i * NB * LD + e;
      static_for<NB>([&](auto mc) {
        constexpr int M = decltype(mc)::value;
        if constexpr (in_part(M)) o[M * LD] = out[M];
      });
    });
  }

  // back to the orthonormal basis (sI: inverse mode scales), mass shift (SHIFT), output; true if a
  // non-finite value was written
  template <bool SHIFT>
  static __device__ __forceinline__ bool store(const R* in, R* out, int e0, int cnt, const R* sI, const R* O,
                                               const R* sGeo, int tid, int nt) {
    bool bad = false;
    for (int t = tid; t < 4 * NB * E; t += nt) {
      const int m = t / E, e = t - m * E;
      if (e >= cnt) continue;
      const size_t g = (size_t)(e0 + e) * 4 * NB + m;
      R v = O[t] * sI[m % NB];
      if (SHIFT && m < 3 * NB) v += sGeo[GEO * e + 7] * in[g];
      bad |= !finite_bits(v);
      out[g] = v;
    }
    return bad;
  }
};

}  // namespace dg
