// Preconditioner assembly at the current linearisation (Sec. 2.3-2.4):
//  * the state-independent linear part of J (viscous and BR2 terms, pressure
//    gradient, continuity) is probed once per handle with unit vectors on the
//    elements of one colour: a distance-1 colouring (no two face neighbours share
//    a colour) for the element diagonal blocks, a distance-2 colouring (no element
//    has two face neighbours of one colour) for the off-diagonal blocks at the
//    degree of level 1 (Sec. 2.4.3: coarse off-diagonal blocks are built at the
//    coarse degree);
//  * the state-dependent part (convective volume term, Riemann face terms) and
//    the mass shift are assembled directly per element at every call;
//  * inherited operators of every coarser level by sub-block extraction
//    (Eq. (GalProj) with a hierarchical orthonormal basis);
//  * LU factors with partial pivoting of all diagonal blocks (element-wise block
//    Jacobi), one block per CTA in shared memory.
// Blocks are stored column-major: block[c * b + r] = G[row r][col c].
#include <algorithm>
#include <vector>

#include "dg_async.h"
#include "dg_internal.h"
#include "dg_pencil.h"

namespace dg {

// ------------------------------------------------ direct state-dependent assembly
// J = J_lin + J_state. J_lin (viscous and BR2 terms, pressure gradient, continuity)
// depends on the mesh only; its blocks are probed once per handle (MODE_LINPART).
// J_state is assembled here per element from the cached linearisation:
//  * convective volume term: -int (u_p u_i)' d_p phi_m with weighted mass matrices
//    U_c[n'][n] = sum_q w_q ubar_c(q) phi_hat_n'(q) phi_hat_n(q) (|K|/8 / s^2 = 1):
//    A[i,m; j,n] = -J_j (D_j^T U_i)[m][n] - delta_ij sum_p J_p (D_p^T U_p)[m][n];
//  * Riemann face terms: with the cached flux Jacobian dF_i/ds_j at the face points
//    and phi_m on a face = P_hat_a(+-1) B2[q][n2(m)] / s, each face adds
//    sign * A4/(s s') P_hat_a(side) P_hat_a'(side') E_ij[n2(m)][n2(n)],
//    E_ij = sum_q w2_q dF_i/ds_j(q) B2[q][n2] B2[q][n2'].
// Diagonal blocks use the own side's columns of the Jacobian; the level-1 off-diagonal
// blocks the other side's, restricted to the coarse modes.
//
// Bound: the bytes of the blocks and of the linear part (240 KB per element at k = 4 over k = 2 in
// FP32), if the instructions stay few. So
//  * E and U come from the same step, plane by plane: a plane of point values against the products
//    of 1D polynomials along its first axis, then along the second, in registers, the pair of 1D
//    exponents fixed at compile time (975 FMA per 15 x 15 matrix instead of 3000);
//  * the two faces of an axis are added before that step: P_hat_a(-1) P_hat_a'(-1) = (-1)^(a+a')
//    P_hat_a(1) P_hat_a'(1), so the faces' difference serves the mode pairs with a + a' even and
//    their sum those with a + a' odd;
//  * the flux Jacobian's zeros are left out: (i, j) couples through axis d only if j is the pressure
//    or d, or if i = j, which leaves 10 of 16 pairs;
//  * one column variable j at a time, so that the matrices take little shared memory (57 KB in FP32 at
//    k = 4) and several elements per SM hide each other's phases; a thread of the output phase
//    keeps one row and loads the linear part kAsmAhead columns at a time.
//  * the next element's Jacobian records and velocity arrive by asynchronous copies while the last column
//    of this one is written, and the linear part is brought to L2 one column variable ahead.
// With every E by direct quadrature and six face terms per entry, FP64 at 12^3 P3 took 1.59 ms, now
// 0.5; FP32 at 24 x 12 x 12 P3 0.61 ms, now 0.37; at 32^3 P4 12.2 ms, now 5.1.
template <int K>
struct PairProducts {
  double v[(K + 1) * (K + 2) / 2][K + 1];
};
// P_hat_a1 P_hat_a2 at the Gauss nodes (ascending), pairs a1 <= a2 at tri(a2) + a1
template <int K>
constexpr PairProducts<K> make_pair_products() {
  PairProducts<K> t{};
  for (int a2 = 0; a2 <= K; ++a2)
    for (int a1 = 0; a1 <= a2; ++a1)
      for (int q = 0; q <= K; ++q) {
        const double x = 2 * q < K ? -gauss_x(K + 1, q) : gauss_x(K + 1, K - q);
        t.v[tri(a2) + a1][q] = leg_scale(a1) * legendre(a1, x) * leg_scale(a2) * legendre(a2, x);
      }
  return t;
}
template <class R, int K>
struct PairTab {
  R v[(K + 1) * (K + 2) / 2][K + 1];
};
template <class R, int K>
constexpr PairTab<R, K> make_pair_tab() {
  constexpr PairProducts<K> p = make_pair_products<K>();
  PairTab<R, K> t{};
  for (int j = 0; j < (K + 1) * (K + 2) / 2; ++j)
    for (int q = 0; q <= K; ++q) t.v[j][q] = R(p.v[j][q]);
  return t;
}
template <class R, int K>
__constant__ PairTab<R, K> pair_tab = make_pair_tab<R, K>();

template <int K, class R = double>
struct AsmSmem {
  static constexpr int NB = nb_of(K), NBM = nb_of(K - 1), N1 = K + 1, NN = N1 * N1, NQ = NN * N1, N2 = tri(K + 1);
  static constexpr int VP = NN | 1, EP = N2 * N2 | 1;  // odd strides of planes and matrices: no bank conflicts
  static constexpr int NT = K == 4 ? 288 : 256;          // threads: whole sets of 4 NB rows
  static constexpr int MATS = 24;                        // matrices of the pressure column, the most at a time
  static constexpr int RAW = 0;                          // [6][4][NN][4] the slots' Jacobian records
  static constexpr int V = RAW + 6 * 16 * NN;            // [2 MATS][NN] weighted point values: own side, other side
  static constexpr int E = V + 2 * MATS * VP;            // [MATS][N2][N2]
  static constexpr int U = E + MATS * EP;                // [3][NBM][NB]
  static constexpr int S = U + 3 * NBM * NB;             // [NB][NB] sum_p J_p (D_p^T U_p)
  static constexpr int PV = S + NB * NB;                 // [2][N1] P_hat_a(+1), P_hat_a(-1)
  static constexpr int PP = PV + 2 * N1;                 // [N2][N1] pair_tab
  static constexpr int PN = PP + N2 * N1;                // [3][NB] P_hat of mode n's exponent along d at +1
  static constexpr int UB = PN + 3 * NB;                 // [3][NQ] the linearisation velocity
  static constexpr int SLOT = UB + 3 * NQ;               // [2 elements][6] scale of the slot's off-diagonal block
  static constexpr int EO = SLOT + 12;                   // [MATS][n2c][n2c] the other side's, for the coarse 2D modes
  __host__ __device__ static constexpr int reals(int n2c) { return EO + MATS * (n2c * n2c | 1); }
  static constexpr int FM = 0;                           // [3][NB] 2D mode of mode n on a face normal to d
  static constexpr int EX = FM + 3 * NB;                 // [3][NB] exponent of mode n along d
  static constexpr int OFF = EX + 3 * NB;                // [3][2][NB] matrix pair and column of mode n, by the row's parity
  static constexpr int SI = OFF + 6 * NB;                // [2 elements][6][2] neighbour (-1: wall), first slot facing it
  static constexpr int INTS = SI + 24;
  __host__ __device__ static constexpr size_t bytes(int n2c) { return sizeof(R) * reals(n2c) + sizeof(int) * INTS; }
};

template <class R>
struct AsmArgs {
  MeshDev M;
  Tables T;
  const R* wvol;       // tables in the assembly precision
  const R* W2;
  const R* pv;
  const R* Dcol_val;
  const R* ubar;       // linearisation cache in the assembly precision
  const R* dFlux;
  const double* Dlin;  // level 0 linear-part diagonal blocks (FP64, probed once)
  R* D;                // level 0 diagonal blocks (output)
  const double* Blin;  // level 1 linear-part off-diagonal blocks (FP64)
  R* Bsr;              // level 1 block rows (output, slots 1..6)
  int nb1;             // modes per variable on level 1 (0: no coarse level)
  double inv_gdt;
};

// Entry (i, j) of the Riemann flux's Jacobian at a face point with normal d, columns of the - side
// (s = 0) or the + side (s = 1), from its 16 stored values (ac_riemann in dg_riemann.h; quad k of the
// point at p + k * stride).
template <class R>
__device__ __forceinline__ R flux_jacobian(const R* p, int stride, int d, int i, int j, int s) {
  if (i == 3 || i == d) {  // du* or dF_n: normal velocity and pressure only
    if (j != 3 && j != d) return R(0);
    return p[(i == d ? stride : 0) + 2 * s + (j == 3)];
  }
  if (j == i) return p[2 * stride + 2 + s];
  if (j != 3 && j != d) return R(0);
  const int t = i == (d == 2 ? 0 : d + 1) ? 0 : 1;
  const R v = p[2 * stride + t] * p[2 * s + (j == 3)];
  return j == 3 ? v : v + p[3 * stride + 2 * t + s];
}

// M[A][B] = sum_{q1, q2} v[q1][q2] B_A B_B(q1, q2) over the 2D modes A, B of degree <= kmax (<= K),
// symmetric, rows of ld; plane(it, v, m, kmax, ld): the plane and matrix of item it < items, false to
// skip it. One thread per item and pair a1 <= a2 of exponents along the first axis. A loop with the
// exponents at run time: unrolled over the pairs at compile time (15 code paths at k = 4, three instances)
// the kernel waited on instruction fetch 60 % of the time.
template <int K, class R, class Plane>
__device__ __forceinline__ void plane_matrices(int items, const R* sPP, int tid, int nt, Plane plane) {
  constexpr int N1 = K + 1;
  for (int w = tid; w < items * tri(N1); w += nt) {
    const int pr = w / items, it = w - pr * items;
    int a2 = 0;
    while (tri(a2 + 1) <= pr) ++a2;
    const int a1 = pr - tri(a2);
    const R* v;
    R* m;
    int kmax, ld;
    if (!plane(it, v, m, kmax, ld)) continue;
    R t[N1];
#pragma unroll
    for (int q2 = 0; q2 < N1; ++q2) t[q2] = R(0);
#pragma unroll
    for (int q = 0; q < N1; ++q) {
      const R pp = sPP[pr * N1 + q];
#pragma unroll
      for (int q2 = 0; q2 < N1; ++q2) t[q2] += pp * v[q * N1 + q2];
    }
    const bool sym = a1 == a2;
    const int n2 = kmax - a2;
    // the 2D modes (a1, b1), (a2, b2)
    for (int b1 = 0, b2 = 0; b1 <= kmax - a1 && b2 <= n2;) {
      const int i = tri(a1 + b1) + b1, j = tri(a2 + b2) + b2;
      const R* pp = sPP + (b1 <= b2 ? tri(b2) + b1 : tri(b1) + b2) * N1;
      R s = R(0);
#pragma unroll
      for (int q = 0; q < N1; ++q) s += pp[q] * t[q];
      m[i * ld + j] = s;
      m[j * ld + i] = s;
      if (++b2 > n2) {
        ++b1;
        b2 = sym ? b1 : 0;
      }
    }
  }
}

constexpr int kAsmAhead = 6;  // columns of the linear part a thread loads at a time

template <int K, class R>
__global__ void __launch_bounds__(AsmSmem<K, R>::NT, sizeof(R) == 4 ? 3 : 2) assemble_state_kernel(AsmArgs<R> a) {
  using L = AsmSmem<K, R>;
  constexpr int NB = L::NB, NBM = L::NBM, N1 = L::N1, NN = L::NN, NQ = L::NQ, N2 = L::N2, VP = L::VP, NN2 = L::EP;
  constexpr int BS = 4 * NB, MATS = L::MATS, nt = L::NT, nw = nt / 32, DW = (K + 1) / 2, TW = Tables::kDw;
  extern __shared__ __align__(16) unsigned char smraw_[];
  R* sm = reinterpret_cast<R*>(smraw_);
  R* sRaw = sm + L::RAW;
  R* sV = sm + L::V;
  R* sE = sm + L::E;
  R* sU = sm + L::U;
  R* sS = sm + L::S;
  R* sPv = sm + L::PV;
  R* sPP = sm + L::PP;
  R* sPn = sm + L::PN;
  R* sUb = sm + L::UB;
  R* sEo = sm + L::EO;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int nb1 = a.nb1, b1 = 4 * nb1;
  int k1 = 0;  // the coarse degree: the graded orderings list the modes of degree <= k1 first
  while (nb1 > 0 && nb_of(k1) < nb1) ++k1;
  const int N2c = nb1 > 0 ? tri(k1 + 1) : 0, NC2 = N2c * N2c | 1;
  int* ism = reinterpret_cast<int*>(sm + L::reals(N2c));
  int* FM = ism + L::FM;
  int* EX = ism + L::EX;
  int* OFF = ism + L::OFF;
  for (int t = tid; t < 3 * NB; t += nt) {
    const int d = t / NB, x = a.T.fa[t], f = a.T.fmap[t];
    FM[t] = f;
    EX[t] = x;
    sPn[t] = a.pv[x];
    OFF[t + d * NB] = (x & 1 ? NN2 : 0) + f;  // row of even exponent
    OFF[t + (d + 1) * NB] = (x & 1 ? 0 : NN2) + f;
  }
  for (int t = tid; t < 2 * N1; t += nt) sPv[t] = a.pv[t];
  for (int t = tid; t < N2 * N1; t += nt) sPP[t] = pair_tab<R, K>.v[t / N1][t % N1];
  __syncthreads();
  // the rows of the output phases: thread -> row (i, m) of every PARTS-th column
  constexpr int PARTS = nt / BS;
  const int row = tid % BS, part = tid / BS, ri = row / NB, rm = row - ri * NB;
  const int parts1 = nb1 > 0 ? nt / b1 : 1, row1 = nb1 > 0 ? tid % b1 : 0, part1 = nb1 > 0 ? tid / b1 : 0;
  const int ri1 = nb1 > 0 ? row1 / nb1 : 0, rm1 = row1 - ri1 * nb1;
  const int qs = nb1 > 0 ? parts1 / nb1 : 0, rs = parts1 - qs * nb1;

  // asynchronous copies of the next element's Jacobian records and velocity, its neighbours and block
  // scales; its linear part goes to L2 one column variable ahead of its use
  auto fetch = [&](int e, int buf) {
    constexpr int CH = NN * (int)sizeof(R);  // 16-byte pieces of a record
    for (int t = tid; t < 6 * CH; t += nt) {
      const int sl = t / CH, c = t - sl * CH, d = sl >> 1, nb = a.M.nbr[(size_t)e * 6 + sl];
      const int f = sl & 1 ? 3 * e + d : (nb >= 0 ? 3 * nb + d : 3 * a.M.ne + a.M.bslot[e]);
      async_16(reinterpret_cast<unsigned char*>(sRaw) + 16 * t,
               reinterpret_cast<const unsigned char*>(a.dFlux + (size_t)f * 16 * NN) + 16 * c);
    }
    for (int t = tid; t < 3 * NQ; t += nt) async_value(sUb + t, a.ubar + (size_t)e * 3 * NQ + t, true);
    const int sl = nt - 1 - tid;
    if (sl < 6) {
      int* SI = ism + L::SI + 12 * buf;
      const int d = sl >> 1, p = a.M.nbr[(size_t)e * 6 + sl];
      int tgt = sl;
      for (int s2 = 0; s2 < sl; ++s2)
        if (a.M.nbr[(size_t)e * 6 + s2] == p) { tgt = s2; break; }
      SI[2 * sl] = p;
      SI[2 * sl + 1] = tgt;
      R sc = R(0);
      if (p >= 0) {
        const ElemGeom g = elem_geom(a.M, e), gp = elem_geom(a.M, p);
        auto h3 = [&](int c) { return c == 0 ? g.h[0] : (c == 1 ? g.h[1] : g.h[2]); };  // no local memory
        sc = R((sl & 1 ? 1.0 : -1.0) * 0.25 * h3((d + 1) % 3) * h3((d + 2) % 3) * g.is * gp.is);
      }
      sm[L::SLOT + 6 * buf + sl] = sc;
    }
  };
  auto prefetch_linear = [&](int e, int j) {
    if (warp != 0 || lane > 6) return;
    if (lane == 6) {
      const double* p = a.Dlin + ((size_t)e * BS + j * NB) * BS;
      prefetch_l2(p, p + NB * BS);
    } else if (nb1 > 0) {
      const double* p = a.Blin + ((size_t)e * 7 + 1 + lane) * b1 * b1 + (size_t)j * nb1 * b1;
      prefetch_l2(p, p + nb1 * b1);
    }
  };
  int buf = 0;
  if ((int)blockIdx.x < a.M.ne) {
    fetch(blockIdx.x, 0);
    prefetch_linear(blockIdx.x, 0);
  }
  for (int e = blockIdx.x; e < a.M.ne; e += gridDim.x, buf ^= 1) {
    const int* SI = ism + L::SI + 12 * buf;
    const R* sScl = sm + L::SLOT + 6 * buf;
    const R* geo = geo_row<R>(a.M, e);
    const R J[3] = {geo[5], geo[6], geo[7]};
    auto jd = [&](int c) { return c == 0 ? J[0] : (c == 1 ? J[1] : J[2]); };  // no local-memory copy
    // weighted entries of column j: own side, the two faces of an axis combined (planes 2 p even, 2 p + 1
    // odd), and the other side's slot by slot. Pairs p of j < 3: (axis j, i = p) for p < 4, then
    // (the other two axes, i = j); of j = 3: (axis p / 4, i = p % 4).
    auto load_column = [&](int j) {
      const int np = j < 3 ? 6 : 12;
      for (int t = tid; t < 3 * np * NN; t += nt) {
        const int w = t / NN, q = t - w * NN;
        const int p = w < np ? w : (w - np) >> 1;
        const int d = j == 3 ? p >> 2 : (p < 4 ? j : (j + p - 3) % 3), i = j == 3 ? p & 3 : (p < 4 ? p : j);
        const R w2 = __ldg(a.W2 + q);
        if (w < np) {
          R v[2];
#pragma unroll
          for (int hi = 0; hi < 2; ++hi) {
            const R* pj = sRaw + ((2 * d + hi) * 4 * NN + q) * 4;
            v[hi] = flux_jacobian(pj, 4 * NN, d, i, j, 1 - hi);
            // at a wall the ghost state (-u_K, p_K) is the element's own: its columns add with
            // sign -1 (velocity) and +1 (pressure)
            if (SI[2 * (2 * d + hi)] < 0) v[hi] += (j == 3 ? R(1) : -R(1)) * flux_jacobian(pj, 4 * NN, d, i, j, hi);
          }
          sV[(2 * p) * VP + q] = w2 * (v[1] - v[0]);
          sV[(2 * p + 1) * VP + q] = w2 * (v[1] + v[0]);
        } else if (nb1 > 0) {
          const int hi = (w - np) & 1, sl = 2 * d + hi;
          sV[(MATS + 2 * p + hi) * VP + q] =
              SI[2 * sl] >= 0 ? w2 * flux_jacobian(sRaw + (sl * 4 * NN + q) * 4, 4 * NN, d, i, j, hi) : R(0);
        }
      }
    };
    async_wait_all();
    __syncthreads();
    // planes of the weighted linearisation velocity
    for (int t = tid; t < 3 * NQ; t += nt) sV[t / NN * VP + t % NN] = __ldg(a.wvol + t % NQ) * sUb[t];
    const bool dup = SI[1] != 0 || SI[3] != 1 || SI[5] != 2 || SI[7] != 3 || SI[9] != 4 || SI[11] != 5;
    const R shift = R(a.inv_gdt * a.M.geo[(size_t)e * kGeo + 11]);
#pragma unroll 1
    for (int j = -1; j < 4; ++j) {  // the volume term's planes, then the column variables
      const int n = j < 0 ? 3 * N1 : (j < 3 ? 12 : 24);
      auto planes = [&](int it, const R*& v, R*& m, int& kmax, int& ld) {
        const bool oth = it >= n;
        const int p = oth ? it - n : it;
        v = sV + (oth ? MATS + p : p) * VP;
        m = oth ? sEo + p * NC2 : sE + p * NN2;
        kmax = oth ? k1 : K;
        ld = oth ? N2c : N2;
        return !oth || nb1 > 0;
      };
      __syncthreads();
      plane_matrices<K, R>(j < 0 ? n : 2 * n, sPP, tid, nt, planes);
      if (j == 0)
        for (int t = tid; t < NB * NB; t += nt) {
          const int m = t / NB, n2 = t - m * NB;
          R s = R(0);
#pragma unroll
          for (int p = 0; p < 3; ++p)
#pragma unroll
            for (int q = 0; q < DW; ++q) {
              const int o = (p * NB + m) * TW + q;
              s += J[p] * __ldg(a.Dcol_val + o) * sU[(p * NBM + __ldg(a.T.Dcol_idx + o)) * NB + n2];
            }
          sS[t] = s;
        }
      __syncthreads();
      const int en = e + gridDim.x;
      if (j < 3) {
        load_column(j + 1);
        if (j >= 0) prefetch_linear(e, j + 1);
      } else if (en < a.M.ne) {
        fetch(en, buf ^ 1);
        prefetch_linear(en, 0);
      }
      if (j < 0) {
        // U_c[n1][n], n1 of degree <= K - 1 (what a derivative reaches), along the planes' normal
        for (int t = tid; t < NBM * NB; t += nt) {
          const int n1 = t / NB, n2 = t - n1 * NB, x1 = EX[n1], x = EX[n2];
          const R* pp = sPP + (x1 <= x ? tri(x) + x1 : tri(x1) + x) * N1;
          const R* Et = sE + FM[n1] * N2 + FM[n2];
#pragma unroll
          for (int c = 0; c < 3; ++c) {
            R u = R(0);
#pragma unroll
            for (int q = 0; q < N1; ++q) u += pp[q] * Et[(c * N1 + q) * NN2];
            sU[c * NBM * NB + t] = u;
          }
        }
        continue;
      }
      if (part < PARTS) {
        const double* Dl = a.Dlin + ((size_t)e * BS + j * NB) * BS + row;
        R* Dout = a.D + ((size_t)e * BS + j * NB) * BS + row;
        // face terms of the row: up to three axes, coefficient J_d P_hat_a(1) and row of a matrix pair
        R fc[3];
        const R* fe[3];
        const R* fp[3];
        const int* fo[3];
#pragma unroll
        for (int x = 0; x < 3; ++x) {
          const int d = j == 3 ? x : (j + x) % 3;
          const int mat = j == 3 ? 8 * x + 2 * ri : (x == 0 ? 2 * ri : 6 + 2 * x);
          fc[x] = jd(d) * sPn[d * NB + rm];
          fe[x] = sE + mat * NN2 + FM[d * NB + rm] * N2;
          fp[x] = sPn + d * NB;
          fo[x] = OFF + (2 * d + (EX[d * NB + rm] & 1)) * NB;
        }
        const bool same = ri == j && j < 3, vol = ri < 3 && j < 3;
        const int nx = j == 3 || same ? 3 : 1;
        const R* uq[DW];
        R uc[DW];
#pragma unroll
        for (int q = 0; q < DW; ++q) {
          const int o = ((vol ? j : 0) * NB + rm) * TW + q;
          uq[q] = sU + ((vol ? ri : 0) * NBM + __ldg(a.T.Dcol_idx + o)) * NB;
          uc[q] = vol ? jd(j) * __ldg(a.Dcol_val + o) : R(0);
        }
        for (int n0 = part; n0 < NB; n0 += kAsmAhead * PARTS) {
          double dl[kAsmAhead];
#pragma unroll
          for (int u = 0; u < kAsmAhead; ++u) {
            const int n = n0 + u * PARTS;
            dl[u] = n < NB ? __ldg(Dl + (size_t)n * BS) : 0.0;
          }
#pragma unroll
          for (int u = 0; u < kAsmAhead; ++u) {
            const int n = n0 + u * PARTS;
            if (n < NB) {
              R v = R(dl[u]);
              if (vol) {
                R cv = R(0);
#pragma unroll
                for (int q = 0; q < DW; ++q) cv += uc[q] * uq[q][n];
                v -= cv;
                if (same) {
                  v -= sS[rm * NB + n];
                  if (n == rm) v += shift;
                }
              }
#pragma unroll
              for (int x = 0; x < 3; ++x)
                if (x < nx) v += fc[x] * fp[x][n] * fe[x][fo[x][n]];
              Dout[(size_t)n * BS] = v;
            }
          }
        }
      }
      // level-1 off-diagonal blocks, coarse modes only: the linear part of the slot plus the Riemann
      // terms of every slot facing the same neighbour, in slot order (a neighbour met on two faces
      // keeps its block at the first slot; the other is zero; a wall slot is zero)
      if (part1 < parts1 && nb1 > 0) {
        const size_t base = (size_t)e * 7 * b1 * b1 + (size_t)j * nb1 * b1 + row1;
        // every parts1-th (slot, column) pair in order, without a division per entry
        int so_l = part1 / nb1, n_l = part1 - so_l * nb1, so_s = so_l, n_s = n_l;
        auto next = [&](int& so, int& n) {
          so += qs;
          n += rs;
          if (n >= nb1) {
            n -= nb1;
            ++so;
          }
        };
        while (so_s < 6) {
          double bl[kAsmAhead];
#pragma unroll
          for (int u = 0; u < kAsmAhead; ++u) {
            bl[u] = so_l < 6 ? __ldg(a.Blin + base + (size_t)(1 + so_l) * b1 * b1 + (size_t)n_l * b1) : 0.0;
            next(so_l, n_l);
          }
#pragma unroll
          for (int u = 0; u < kAsmAhead; ++u) {
            const int so = so_s, n = n_s;
            if (so >= 6) break;
            next(so_s, n_s);
            R v = R(0);
            if (SI[2 * so] >= 0 && SI[2 * so + 1] == so) {
              v = R(bl[u]);
              for (int sl = so; sl < (dup ? 6 : so + 1); ++sl) {
                if (SI[2 * sl] < 0 || SI[2 * sl + 1] != so) continue;
                const int d = sl >> 1, hi = sl & 1, dj = d - j + (d < j ? 3 : 0);
                if (j < 3 && d != j && ri1 != j) continue;  // no coupling through this axis
                const int mat = j == 3 ? 2 * (4 * d + ri1) + hi : (d == j ? 2 * ri1 + hi : 6 + 2 * dj + hi);
                v += sScl[sl] * sPv[(1 - hi) * N1 + EX[d * NB + rm1]] * sPv[hi * N1 + EX[d * NB + n]] *
                     sEo[mat * NC2 + FM[d * NB + rm1] * N2c + FM[d * NB + n]];
              }
            }
            a.Bsr[base + (size_t)(1 + so) * b1 * b1 + (size_t)n * b1] = v;
          }
        }
      }
    }
  }
}

template <int K, class R>
static int launch_assemble_state(Handle* h, const AsmArgs<R>& a, cudaStream_t st) {
  // the coarse face matrices are sized for the handle's level-1 degree
  const int n2c = a.nb1 > 0 ? tri(h->lev[1].k + 1) : 0, threads = AsmSmem<K, R>::NT;
  const size_t smem = AsmSmem<K, R>::bytes(n2c);
  DG_CUDA(h, cudaFuncSetAttribute(assemble_state_kernel<K, R>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  int per_sm = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, assemble_state_kernel<K, R>, threads, smem) != cudaSuccess ||
      per_sm < 1)
    per_sm = 1;
  const int grid = std::min(h->ne, h->nsm * per_sm);
  assemble_state_kernel<K, R><<<grid, threads, smem, st>>>(a);
  DG_LAUNCH_CHECK(h);
  return DG_OK;
}

static std::vector<int> greedy_colouring(const Handle* h, int dist) {
  const int ne = h->ne;
  const std::vector<int>& nb6 = h->nbr_host;
  std::vector<int> col(ne, -1);
  if (dist == 2 && h->nprob == 1 && h->n[0] % 8 == 0 && h->n[1] % 8 == 0 && h->n[2] % 8 == 0) {
    // (i + 2j + 3k) mod 8: the six neighbour offsets +-1, +-2, +-3 are distinct and non-zero mod 8,
    // so no element shares a colour with a neighbour or with a neighbour's neighbour
    for (int e = 0; e < ne; ++e) {
      const int i = e % h->n[0], j = (e / h->n[0]) % h->n[1], k = e / (h->n[0] * h->n[1]);
      col[e] = (i + 2 * j + 3 * k) % 8;
    }
    return col;
  }
  std::vector<int> mark(64, -1);
  for (int e = 0; e < ne; ++e) {
    std::vector<int> around;
    for (int f = 0; f < 6; ++f) {
      const int p = nb6[e * 6 + f];
      if (p < 0) continue;  // a wall
      around.push_back(p);
      if (dist >= 2)
        for (int g = 0; g < 6; ++g)
          if (nb6[p * 6 + g] >= 0) around.push_back(nb6[p * 6 + g]);
    }
    for (int p : around)
      if (p != e && col[p] >= 0) mark[col[p]] = e;
    int c = 0;
    while (mark[c] == e) ++c;
    col[e] = c;
  }
  return col;
}

__global__ void probe_kernel(long long n, int b, const int* colour, int c, int j, double* v) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const long long e = i / b;
    const int r = (int)(i - e * b);
    v[i] = (colour[e] == c && r == j) ? 1.0 : 0.0;
  }
}

// Dblk[e][j][r] = out[e][r] for elements of colour c.
__global__ void scatter_diag_kernel(int ne, int b, const int* colour, int c, int j, const double* out, double* D) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < (long long)ne * b;
       i += (long long)gridDim.x * blockDim.x) {
    const long long e = i / b;
    const int r = (int)(i - e * b);
    if (colour[e] == c) D[(e * b + j) * b + r] = out[e * b + r];
  }
}

// For every element p and face slot f whose neighbour e = nbr[p][f] has colour c
// (and f is the first slot of p facing e): Bsr1[p][1+f][jc][rc] = out[p][fine row of rc].
__global__ void scatter_offdiag_kernel(int ne, int nb0, int nb1, const int* nbr, const int* colour, int c, int jc,
                                       const double* out, double* Bsr) {
  const int b1 = 4 * nb1;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < (long long)ne * 6 * b1;
       i += (long long)gridDim.x * blockDim.x) {
    const long long p = i / (6 * b1);
    const int rem = (int)(i - p * 6 * b1), f = rem / b1, rc = rem - f * b1;
    const int e = nbr[p * 6 + f];
    if (e < 0 || colour[e] != c) continue;
    bool first = true;
    for (int g = 0; g < f; ++g)
      if (nbr[p * 6 + g] == e) first = false;
    if (!first) continue;
    const int var = rc / nb1, m = rc - var * nb1;
    Bsr[(((p * 7 + 1 + f) * (long long)b1) + jc) * b1 + rc] = out[(p * 4 + var) * nb0 + m];
  }
}

// Row-block probing: for every element p, slot 0 (p itself, when p has colour c) and each face
// slot f whose neighbour e = nbr[p][f] has colour c (first slot facing e only):
// A[p][slot][jc][rc] += sign * out[p][fine row of rc] (level-1 modes nb1 of nb0).
__global__ void scatter_rows_kernel(int ne, int nb0, int nb1, const int* nbr, const int* colour, int c, int jc,
                                    const double* out, double sign, double* A) {
  const int b1 = 4 * nb1;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < (long long)ne * 7 * b1;
       i += (long long)gridDim.x * blockDim.x) {
    const long long p = i / (7 * b1);
    const int rem = (int)(i - p * 7 * b1), s = rem / b1, rc = rem - s * b1;
    const int e = s == 0 ? (int)p : nbr[p * 6 + s - 1];
    if (e < 0 || colour[e] != c) continue;
    if (s > 0) {
      bool first = true;
      for (int g = 0; g < s - 1; ++g)
        if (nbr[p * 6 + g] == e) first = false;
      if (!first || e == (int)p) continue;
    }
    const int var = rc / nb1, m = rc - var * nb1;
    A[(((p * 7 + s) * (long long)b1) + jc) * b1 + rc] += sign * out[(p * 4 + var) * nb0 + m];
  }
}

// Inherited coarse blocks (Eq. (GalProj) with a hierarchical orthonormal basis: the leading
// sub-block of every variable pair), with the rescaling of Appendix A: for the slots
// s = blockIdx.y of every element block, dst = sub(src) [+ coef * sub(stb)], where stb holds the
// level-1 stabilisation blocks (nb1 modes per variable) and src the finer blocks (nbs modes);
// dst2, if given, receives a second copy. src and dst may be the same blocks (an in-place add).
// One CTA row per slot, 32-bit index arithmetic within a block, arithmetic in R.
template <class R>
__global__ void inherit_kernel(int nblocks, int nbs, const R* src, long long src_blk, long long src_slot, int nbd,
                               R* dst, long long dst_blk, long long dst_slot, R* dst2, long long dst2_blk,
                               const R* __restrict__ stb, long long stb_blk, long long stb_slot, int nb1, R coef) {
  const int bs = 4 * nbs, bd = 4 * nbd, b1 = 4 * nb1, sl = blockIdx.y;
  for (int blk = blockIdx.x; blk < nblocks; blk += gridDim.x) {
    const R* sb = src + blk * src_blk + sl * src_slot;
    const R* tb = stb ? stb + blk * stb_blk + sl * stb_slot : nullptr;
    R* db = dst + blk * dst_blk + sl * dst_slot;
    R* d2 = dst2 ? dst2 + blk * dst2_blk : nullptr;
    for (int t = threadIdx.x; t < bd * bd; t += blockDim.x) {
      const int c = t / bd, r = t - c * bd;
      const int cv = c / nbd, cm = c - cv * nbd, rv = r / nbd, rm = r - rv * nbd;
      R v = sb[(cv * nbs + cm) * bs + rv * nbs + rm];
      if (tb) v += coef * tb[(cv * nb1 + cm) * b1 + rv * nb1 + rm];
      db[t] = v;
      if (d2) d2[t] = v;
    }
  }
}

// In-place LU factorisation with partial (row) pivoting of one b x b block per CTA in
// shared memory (row-major, padded leading dimension). Output, column-major per block:
// the unit-lower L below the diagonal, U with its rows scaled by 1/U_kk above it, and 1/U_kk on the
// diagonal (backward substitution then needs no division or product per step); and the row
// permutation pi (row i of P A is row pi[i] of A).
template <class R>
__global__ void __launch_bounds__(256) lu_factor_kernel(int nblk, int b, const R* in, R* out, int* perm,
                                                       unsigned* status) {
  extern __shared__ __align__(16) unsigned char smraw_[];
  R* sm = reinterpret_cast<R*>(smraw_);
  const int LD = b + 1;
  R* A = sm;                               // [b][LD]
  int* piv = reinterpret_cast<int*>(A + b * LD);  // [b] row swapped with k at step k
  __shared__ int s_piv;
  const int tid = threadIdx.x, nt = blockDim.x, warp = tid >> 5, lane = tid & 31, nw = nt >> 5;
  for (int blk = blockIdx.x; blk < nblk; blk += gridDim.x) {
    const R* src = in + (size_t)blk * b * b;
    for (int t = tid; t < b * b; t += nt) {
      const int c = t / b, r = t - c * b;
      A[r * LD + c] = src[t];
    }
    __syncthreads();
    for (int k = 0; k < b; ++k) {
      if (warp == 0) {
        R best = R(-1);
        int bi = k;
        for (int i = k + lane; i < b; i += 32) {
          const R v = fabs(A[i * LD + k]);
          if (v > best) { best = v; bi = i; }
        }
        for (int off = 16; off > 0; off >>= 1) {
          const R ov = __shfl_down_sync(0xffffffffu, best, off);
          const int oi = __shfl_down_sync(0xffffffffu, bi, off);
          if (ov > best || (ov == best && oi < bi)) { best = ov; bi = oi; }
        }
        if (lane == 0) {
          s_piv = bi;
          piv[k] = bi;
          if (!(best > R(0)) && status) atomicOr(status, (unsigned)DG_STATUS_NONFINITE);
        }
      }
      __syncthreads();
      const int p = s_piv;
      if (p != k)
        for (int j = tid; j < b; j += nt) {
          const R t = A[k * LD + j];
          A[k * LD + j] = A[p * LD + j];
          A[p * LD + j] = t;
        }
      __syncthreads();
      const R rk = R(1) / A[k * LD + k];
      for (int i = k + 1 + tid; i < b; i += nt) A[i * LD + k] *= rk;
      __syncthreads();
      // trailing update: warp w takes rows k+1+w, k+1+w+nw, ...; lanes take the columns
      for (int i = k + 1 + warp; i < b; i += nw) {
        const R l = A[i * LD + k];
        R* Ai = A + i * LD;
        const R* Ak = A + k * LD;
        for (int j = k + 1 + lane; j < b; j += 32) Ai[j] = fma(-l, Ak[j], Ai[j]);
      }
      if (tid == 0) A[k * LD + k] = rk;
      __syncthreads();
    }
    R* dst = out + (size_t)blk * b * b;
    for (int t = tid; t < b * b; t += nt) {
      const int c = t / b, r = t - c * b;
      dst[t] = r < c ? A[r * LD + c] * A[r * LD + r] : A[r * LD + c];
    }
    if (tid == 0) {
      // compose the swaps into pi: apply them in order to the identity
      int* pi = perm + (size_t)blk * b;
      for (int i = 0; i < b; ++i) pi[i] = i;
      for (int kk = 0; kk < b; ++kk) {
        const int q = piv[kk];
        const int t = pi[kk];
        pi[kk] = pi[q];
        pi[q] = t;
      }
    }
    __syncthreads();
  }
}

template <class R>
static int factor_blocks(Handle* h, int nblk, int b, const R* in, R* out, int* perm, cudaStream_t st) {
  const size_t smem = sizeof(R) * (size_t)b * (b + 1) + sizeof(int) * b;
  DG_CUDA(h, cudaFuncSetAttribute(lu_factor_kernel<R>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  int per_sm = (int)((220 * 1024) / smem);
  if (per_sm < 1) per_sm = 1;
  if (per_sm > 8) per_sm = 8;
  int grid = h->nsm * per_sm;
  if (grid > nblk) grid = nblk;
  lu_factor_kernel<R><<<grid, 256, smem, st>>>(nblk, b, in, out, perm, h->status + 2);
  DG_LAUNCH_CHECK(h);
  return DG_OK;
}

// Blocks of the state-independent linear part of J (viscous and BR2 terms, pressure
// gradient, continuity), probed once per handle: element diagonal blocks on level 0 and
// the level-1 off-diagonal blocks.
static int probe_linear_part(Handle* h, cudaStream_t st) {
  const int ne = h->ne;
  Level& L0 = h->lev[0];
  const int b0 = L0.b;
  const int grid = h->nsm * 8;
  int rc;
  if (!h->colour) DG_CUDA(h, cudaMalloc((void**)&h->colour, sizeof(int) * ne));
  int* dcol = h->colour;
  double* probe = L0.t0;
  double* out = L0.t1;
  const std::vector<int> c1 = greedy_colouring(h, 1);
  const int nc1 = *std::max_element(c1.begin(), c1.end()) + 1;
  DG_CUDA(h, cudaMemcpyAsync(dcol, c1.data(), sizeof(int) * ne, cudaMemcpyHostToDevice, st));
  for (int c = 0; c < nc1; ++c)
    for (int j = 0; j < b0; ++j) {
      probe_kernel<<<grid, 256, 0, st>>>(L0.n, b0, dcol, c, j, probe);
      DG_LAUNCH_CHECK(h);
      if ((rc = op_linear_part(h, probe, out, st))) return rc;
      scatter_diag_kernel<<<grid, 256, 0, st>>>(ne, b0, dcol, c, j, out, L0.Dlin);
      DG_LAUNCH_CHECK(h);
    }
  if (h->nlev > 1) {
    Level& L1 = h->lev[1];
    const int b1 = L1.b;
    DG_CUDA(h, cudaMemsetAsync(L1.Blin, 0, sizeof(double) * (size_t)b1 * b1 * 7 * ne, st));
    const std::vector<int> c2 = greedy_colouring(h, 2);
    const int nc2 = *std::max_element(c2.begin(), c2.end()) + 1;
    DG_CUDA(h, cudaMemcpyAsync(dcol, c2.data(), sizeof(int) * ne, cudaMemcpyHostToDevice, st));
    for (int c = 0; c < nc2; ++c)
      for (int jc = 0; jc < b1; ++jc) {
        const int jf = (jc / L1.nb) * L0.nb + jc % L1.nb;
        probe_kernel<<<grid, 256, 0, st>>>(L0.n, b0, dcol, c, jf, probe);
        DG_LAUNCH_CHECK(h);
        if ((rc = op_linear_part(h, probe, out, st))) return rc;
        scatter_offdiag_kernel<<<grid, 256, 0, st>>>(ne, L0.nb, L1.nb, h->nbr, dcol, c, jc, out, L1.Blin);
        DG_LAUNCH_CHECK(h);
      }
  }
  return DG_OK;
}

// The stabilisation part of the level-1 block rows, G(eta) - G(0) probed with the linear part
// (the eta term is linear and state independent), distance-2 colouring.
static int probe_stb(Handle* h, cudaStream_t st) {
  const int ne = h->ne;
  Level& L0 = h->lev[0];
  Level& L1 = h->lev[1];
  const int b0 = L0.b, b1 = L1.b;
  const int grid = h->nsm * 8;
  int rc;
  if (!h->stb1) DG_CUDA(h, cudaMalloc((void**)&h->stb1, sizeof(double) * (size_t)b1 * b1 * 7 * ne));
  DG_CUDA(h, cudaMemsetAsync(h->stb1, 0, sizeof(double) * (size_t)b1 * b1 * 7 * ne, st));
  if (!h->colour) DG_CUDA(h, cudaMalloc((void**)&h->colour, sizeof(int) * ne));
  int* dcol = h->colour;
  double* probe = L0.t0;
  double* out = L0.t1;
  const std::vector<int> c2 = greedy_colouring(h, 2);
  const int nc2 = *std::max_element(c2.begin(), c2.end()) + 1;
  DG_CUDA(h, cudaMemcpyAsync(dcol, c2.data(), sizeof(int) * ne, cudaMemcpyHostToDevice, st));
  const double eta = h->p.eta;
  for (int pass = 0; pass < 2; ++pass) {
    h->p.eta = pass == 0 ? eta : 0.0;
    for (int c = 0; c < nc2; ++c)
      for (int jc = 0; jc < b1; ++jc) {
        const int jf = (jc / L1.nb) * L0.nb + jc % L1.nb;
        probe_kernel<<<grid, 256, 0, st>>>(L0.n, b0, dcol, c, jf, probe);
        DG_LAUNCH_CHECK(h);
        if ((rc = op_linear_part(h, probe, out, st))) { h->p.eta = eta; return rc; }
        scatter_rows_kernel<<<grid, 256, 0, st>>>(ne, L0.nb, L1.nb, h->nbr, dcol, c, jc, out,
                                                  pass == 0 ? 1.0 : -1.0, h->stb1);
        DG_LAUNCH_CHECK(h);
      }
  }
  h->p.eta = eta;
  return DG_OK;
}

static int alloc_fp32_levels(Handle* h) {
  for (int l = 0; l < h->nlev; ++l) {
    Level& L = h->lev[l];
    const size_t nbb = (size_t)h->ne * L.b * L.b;
    if (!L.LUf) DG_CUDA(h, cudaMalloc((void**)&L.LUf, sizeof(float) * nbb));
    if (!L.t0f) DG_CUDA(h, cudaMalloc((void**)&L.t0f, sizeof(float) * L.n));
    if (!L.t1f) DG_CUDA(h, cudaMalloc((void**)&L.t1f, sizeof(float) * L.n));
    if (!L.t2f) DG_CUDA(h, cudaMalloc((void**)&L.t2f, sizeof(float) * L.n));
    if (l >= 1 && !L.Bsrf) DG_CUDA(h, cudaMalloc((void**)&L.Bsrf, sizeof(float) * nbb * 7));
    if (!L.perm) DG_CUDA(h, cudaMalloc((void**)&L.perm, sizeof(int) * (size_t)h->ne * L.b));
  }
  return DG_OK;
}

template <class R>
static int assemble_levels(Handle* h, const AsmArgs<R>& a, R* const* Dlev, R* const* Bsrlev, const R* stb,
                           cudaStream_t st) {
  const int ne = h->ne;
  const int grid = h->nsm * 8;
  int rc;
  switch (h->tab.k) {
    case 1: rc = launch_assemble_state<1, R>(h, a, st); break;
    case 2: rc = launch_assemble_state<2, R>(h, a, st); break;
    case 3: rc = launch_assemble_state<3, R>(h, a, st); break;
    case 4: rc = launch_assemble_state<4, R>(h, a, st); break;
    default: rc = fail(h, DG_ERR_ARG, "unsupported degree");
  }
  if (rc) return rc;
  const Level& L0 = h->lev[0];
  const int b0 = L0.b;
  // coarse levels: inherited sub-blocks (taken before the fine blocks are factored in place);
  // with the rescaling of Appendix A, the stabilisation part of level l is weighted by S_0^l
  const int k0 = L0.k, nb1 = h->nlev > 1 ? h->lev[1].nb : 0, b1 = 4 * nb1;
  const R* sb = h->stb_rescale ? stb : nullptr;
  const long long s1 = (long long)b1 * b1;
  double s_prev = 1.0;
  for (int l = 1; l < h->nlev; ++l) {
    Level& L = h->lev[l];
    const long long bb = (long long)L.b * L.b;
    const double S = (double)(L.k * (L.k + 3)) / (double)(k0 * (k0 + 3));
    // diagonal: sub(D_0) [+ (S - 1) sub(stabilisation slot 0)], also slot 0 of the block row
    inherit_kernel<R><<<dim3(grid, 1), 256, 0, st>>>(ne, L0.nb, Dlev[0], (long long)b0 * b0, 0, L.nb, Dlev[l], bb, 0,
                                                   Bsrlev[l], bb * 7, sb, s1 * 7, s1, nb1, R(S - 1.0));
    DG_LAUNCH_CHECK(h);
    // off-diagonal slots: level 1's come from the state assembly (the add is in place), level
    // l >= 2 inherits level l - 1's; level 1 carries S - 1, level l >= 2 adds S - s_prev
    if (l >= 2 || sb) {
      const Level& P = h->lev[l == 1 ? 1 : l - 1];
      const long long pbb = (long long)P.b * P.b;
      inherit_kernel<R><<<dim3(grid, 6), 256, 0, st>>>(ne, P.nb, Bsrlev[l == 1 ? 1 : l - 1] + pbb, pbb * 7, pbb,
                                                     L.nb, Bsrlev[l] + bb, bb * 7, bb, nullptr, 0,
                                                     sb ? sb + s1 : nullptr, s1 * 7, s1, nb1,
                                                     R(l == 1 ? S - 1.0 : S - s_prev));
      DG_LAUNCH_CHECK(h);
    }
    s_prev = S;
  }
  return DG_OK;
}

__global__ void narrow_f32_kernel(long long n, const double* __restrict__ x, float* __restrict__ y) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    y[i] = (float)x[i];
}

__global__ void or_bits_kernel(unsigned* status, unsigned bits) { atomicOr(status, bits); }

int assemble_all(Handle* h, int precision, cudaStream_t st) {
  const int ne = h->ne;
  Level& L0 = h->lev[0];
  int rc;
  DG_CUDA(h, cudaMemsetAsync(h->status + 2, 0, sizeof(unsigned), st));  // this assembly's own status word
  // the linear part (FP64, mesh only) and the FP64 fine diagonal-block buffer it lives next to
  if (!L0.Dlin) DG_CUDA(h, cudaMalloc((void**)&L0.Dlin, sizeof(double) * (size_t)L0.b * L0.b * ne));
  if (h->nlev > 1 && !h->lev[1].Blin) {
    const size_t nbl = sizeof(double) * (size_t)h->lev[1].b * h->lev[1].b * 7 * ne;
    DG_CUDA(h, cudaMalloc((void**)&h->lev[1].Blin, nbl));
    DG_CUDA(h, cudaMemsetAsync(h->lev[1].Blin, 0, nbl, st));  // slots across a wall stay zero
  }
  if (!h->linpart_ready) {
    if ((rc = probe_linear_part(h, st))) return rc;
    h->linpart_ready = true;
  }
  if (h->stb_rescale && !h->stb_ready) {
    if ((rc = probe_stb(h, st))) return rc;
    h->stb_ready = true;
  }
  if (precision == DG_PRECOND_FP64) {
    for (int l = 0; l < h->nlev; ++l) {
      Level& L = h->lev[l];
      const size_t bb = (size_t)L.b * L.b;
      if (!L.Dblk) DG_CUDA(h, cudaMalloc((void**)&L.Dblk, sizeof(double) * bb * ne));
      if (!L.Dinv) DG_CUDA(h, cudaMalloc((void**)&L.Dinv, sizeof(double) * bb * ne));
      if (l >= 1 && !L.Bsr) DG_CUDA(h, cudaMalloc((void**)&L.Bsr, sizeof(double) * bb * 7 * ne));
      if (!L.perm) DG_CUDA(h, cudaMalloc((void**)&L.perm, sizeof(int) * (size_t)ne * L.b));
    }
    AsmArgs<double> a;
    a.M = mesh_dev(h);
    a.T = h->tab;
    a.wvol = h->tab.wvol; a.W2 = h->tab.W2; a.pv = h->tab.pv;
    a.Dcol_val = h->tab.Dcol_val;
    a.ubar = h->ubar;
    a.dFlux = h->dFlux;
    a.Dlin = L0.Dlin;
    a.D = L0.Dblk;
    a.Blin = h->nlev > 1 ? h->lev[1].Blin : nullptr;
    a.Bsr = h->nlev > 1 ? h->lev[1].Bsr : nullptr;
    a.nb1 = h->nlev > 1 ? h->lev[1].nb : 0;
    a.inv_gdt = h->inv_gdt;
    double* Dl[DG_MAX_LEVELS];
    double* Bl[DG_MAX_LEVELS];
    for (int l = 0; l < h->nlev; ++l) { Dl[l] = h->lev[l].Dblk; Bl[l] = h->lev[l].Bsr; }
    if ((rc = assemble_levels<double>(h, a, Dl, Bl, h->stb1, st))) return rc;
    for (int l = 0; l < h->nlev; ++l) {
      Level& L = h->lev[l];
      if ((rc = factor_blocks<double>(h, ne, L.b, L.Dblk, L.Dinv, L.perm, st))) return rc;
    }
  } else {
    if ((rc = alloc_fp32_levels(h))) return rc;
    if ((rc = prepare_lin_fp32(h, st))) return rc;
    AsmArgs<float> a;
    const TablesF& F = h->tabf;
    a.M = mesh_dev(h);
    a.T = h->tab;
    a.wvol = F.wvol; a.W2 = F.W2; a.pv = F.pv; a.Dcol_val = F.Dcol_val;
    a.ubar = h->ubar_f;
    a.dFlux = h->dFlux_f;
    a.Dlin = L0.Dlin;
    a.D = L0.LUf;
    a.Blin = h->nlev > 1 ? h->lev[1].Blin : nullptr;
    a.Bsr = h->nlev > 1 ? h->lev[1].Bsrf : nullptr;
    a.nb1 = h->nlev > 1 ? h->lev[1].nb : 0;
    a.inv_gdt = h->inv_gdt;
    float* Dl[DG_MAX_LEVELS];
    float* Bl[DG_MAX_LEVELS];
    for (int l = 0; l < h->nlev; ++l) { Dl[l] = h->lev[l].LUf; Bl[l] = h->lev[l].Bsrf; }
    if (h->stb_rescale && !h->stb1f) {  // an FP32 copy of the stabilisation blocks (fixed per handle)
      const long long n = 7ll * h->lev[1].b * h->lev[1].b * ne;
      DG_CUDA(h, cudaMalloc((void**)&h->stb1f, sizeof(float) * n));
      narrow_f32_kernel<<<h->nsm * 8, 256, 0, st>>>(n, h->stb1, h->stb1f);
      DG_LAUNCH_CHECK(h);
    }
    if ((rc = assemble_levels<float>(h, a, Dl, Bl, h->stb1f, st))) return rc;
    if ((rc = invert_levels_f32(h, st, h->status + 2))) return rc;  // the FP32 smoother applies explicit inverses
  }
  // the verdict on this assembly's own status word (flags of earlier calls do not count); its
  // bits also go to the handle's word, which dg_get_status reads
  DG_CUDA(h, cudaStreamSynchronize(st));
  unsigned s = 0;
  DG_CUDA(h, cudaMemcpy(&s, h->status + 2, sizeof(unsigned), cudaMemcpyDeviceToHost));
  if (s) {
    or_bits_kernel<<<1, 1, 0, st>>>(h->status, s);
    DG_LAUNCH_CHECK(h);
  }
  if (s & DG_STATUS_NONFINITE) return fail(h, DG_ERR_NONFINITE, "singular or non-finite element block");
  return DG_OK;
}

}  // namespace dg
