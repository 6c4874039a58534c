// Building blocks of the matrix-free operator kernels: 1D transforms of pencils of modal
// coefficients, with compile-time tables.
//
// The kernels work on coefficients of plain (unnormalised) Legendre products L_a L_b L_c, scaled
// once where they are loaded: c' = s_a s_b s_c c with s_n = sqrt((2n+1)/2), since the orthonormal
// basis is P_hat_n = s_n L_n. In that basis
//  * traces at xi = +-1 are sums with signs (L_a(+-1) = (+-1)^a);
//  * derivatives are (2a+1) times a sum over every second coefficient
//    (L_n' = sum of (2a+1) L_a over a = n-1, n-3, ...);
//  * L_0 = 1, and the Gauss nodes are symmetric, so a pencil of n coefficients is evaluated at (or
//    projected from) the nodes through its even and odd parts: 14 operations instead of 25 for
//    n = 5, fewer for the shorter pencils of the total-degree basis.
// That matters because GB300's FP64 pipe (2 FMA per clock and SM; a warp instruction holds it for
// 16 clocks) bounds the FP64 passes, whatever the number of threads, and because instruction
// issue bounds the FP32 passes.
#pragma once

#include <cuda_runtime.h>

#include <type_traits>

#include "dg_internal.h"

namespace dg {

__host__ __device__ constexpr int tri(int n) { return n * (n + 1) / 2; }
__host__ __device__ constexpr int tet(int n) { return n * (n + 1) * (n + 2) / 6; }

// Gauss-Legendre rule with n1 points: |x| and weight of the node pair h (h = 0 the outermost);
// h = n1 / 2 is the centre node of an odd rule.
constexpr double gauss_x(int n1, int h) {
  return n1 == 2 ? 0.57735026918962576451
       : n1 == 3 ? (h == 0 ? 0.77459666924148337704 : 0.0)
       : n1 == 4 ? (h == 0 ? 0.86113631159405257522 : 0.33998104358485626480)
                 : (h == 0 ? 0.90617984593866399280 : (h == 1 ? 0.53846931010568309104 : 0.0));
}
constexpr double gauss_w(int n1, int h) {
  return n1 == 2 ? 1.0
       : n1 == 3 ? (h == 0 ? 0.55555555555555555556 : 0.88888888888888888889)
       : n1 == 4 ? (h == 0 ? 0.34785484513745385737 : 0.65214515486254614263)
                 : (h == 0 ? 0.23692688505618908751 : (h == 1 ? 0.47862867049936646804 : 0.56888888888888888889));
}
constexpr double legendre(int n, double x) {
  return n == 0 ? 1.0 : n == 1 ? x : n == 2 ? 1.5 * x * x - 0.5 : n == 3 ? (2.5 * x * x - 1.5) * x
                                     : (4.375 * x * x - 3.75) * x * x + 0.375;
}
// s_n = sqrt((2n+1)/2)
constexpr double leg_scale(int n) {
  return n == 0 ? 0.70710678118654752440 : n == 1 ? 1.22474487139158904910 : n == 2 ? 1.58113883008418966600
       : n == 3 ? 1.87082869338697069279 : 2.12132034355964257320;
}

// 1D tables of degree K: L[h][n] = L_n(x_h) at the positive node of pair h (and the centre), and
// P[h][n] = (2n+1)/2 w_h L_n(x_h), which turns point values into coefficients.
template <class R, int K>
struct PencilTab {
  R L[K / 2 + 1][K + 1];
  R P[K / 2 + 1][K + 1];
  R P2[K / 2 + 1][K + 1];  // 2 P
};
template <class R, int K>
constexpr PencilTab<R, K> make_pencil_tab() {
  PencilTab<R, K> t{};
  for (int h = 0; h < (K + 2) / 2; ++h)
    for (int n = 0; n <= K; ++n) {
      const double l = legendre(n, gauss_x(K + 1, h)), p = 0.5 * (2 * n + 1) * gauss_w(K + 1, h) * l;
      t.L[h][n] = R(l);
      t.P[h][n] = R(p);
      t.P2[h][n] = R(2.0 * p);
    }
  return t;
}
// constant memory, indexed at compile time: the tables are operands of the FMAs, not registers
template <class R, int K>
__constant__ PencilTab<R, K> pencil_tab = make_pencil_tab<R, K>();

// compile-time loop: f(integral_constant 0), ..., f(integral_constant N - 1)
template <class F, int... I>
__device__ __forceinline__ void static_for_(F& f, std::integer_sequence<int, I...>) {
  (f(std::integral_constant<int, I>{}), ...);
}
template <int N, class F>
__device__ __forceinline__ void static_for(F f) {
  static_for_(f, std::make_integer_sequence<int, N>{});
}

// Modes are ordered by degree, then by the x exponent descending, then by the y exponent descending;
// the 2D modes (b, c) of a face by degree, then by b descending.
__host__ __device__ constexpr int mode_exp(int m, int axis) {
  for (int g = 0;; ++g)
    for (int a = g; a >= 0; --a)
      for (int b = g - a; b >= 0; --b, --m)
        if (m == 0) return axis == 0 ? a : (axis == 1 ? b : g - a - b);
}
__host__ __device__ constexpr int mode_at(int a, int b, int c) {  // exponents along x, y, z
  return tet(a + b + c) + tri(b + c) + c;
}
// mode with exponent a along axis d, b along (d+1)%3 and c along (d+2)%3
__host__ __device__ constexpr int mode_along(int d, int a, int b, int c) {
  return d == 0 ? mode_at(a, b, c) : (d == 1 ? mode_at(c, a, b) : mode_at(b, c, a));
}
// degree of 2D mode j
__host__ __device__ constexpr int face_degree(int j) {
  int g = 0;
  while (tri(g + 1) <= j) ++g;
  return g;
}

// scale s_m of every 3D mode of degree K and its inverse, in mode order, in the kernel's precision
// (a conversion from FP64 at run time would go through GB300's FP64 pipe)
template <class R, int K>
struct ModeScale {
  R s[nb_of(K)], inv[nb_of(K)];
};
template <class R, int K>
constexpr ModeScale<R, K> make_mode_scale() {
  ModeScale<R, K> t{};
  for (int m = 0; m < nb_of(K); ++m) {
    const double s = leg_scale(mode_exp(m, 0)) * leg_scale(mode_exp(m, 1)) * leg_scale(mode_exp(m, 2));
    t.s[m] = R(s);
    t.inv[m] = R(1.0 / s);
  }
  return t;
}
template <class R, int K>
__constant__ ModeScale<R, K> mode_scale = make_mode_scale<R, K>();

// c[0..N) -> values at the K + 1 Gauss nodes (ascending)
template <int K, int N, class R>
__device__ __forceinline__ void interp_pencil(const R (&c)[N], R (&v)[K + 1]) {
#pragma unroll
  for (int h = 0; h < (K + 1) / 2; ++h) {
    R ev = c[0];
#pragma unroll
    for (int n = 2; n < N; n += 2) ev += pencil_tab<R, K>.L[h][n] * c[n];
    if constexpr (N == 1) {
      v[h] = ev;
      v[K - h] = ev;
    } else if constexpr (N <= 3) {
      v[K - h] = ev + pencil_tab<R, K>.L[h][1] * c[1];
      v[h] = ev - pencil_tab<R, K>.L[h][1] * c[1];
    } else {
      const R od = pencil_tab<R, K>.L[h][1] * c[1] + pencil_tab<R, K>.L[h][3] * c[3];
      v[K - h] = ev + od;
      v[h] = ev - od;
    }
  }
  if constexpr (K % 2 == 0) {
    R ev = c[0];
#pragma unroll
    for (int n = 2; n < N; n += 2) ev += pencil_tab<R, K>.L[K / 2][n] * c[n];
    v[K / 2] = ev;
  }
}

// values at the K + 1 nodes -> the first N coefficients: o = projection (ACC = 0), or
// o -= projection (ACC = -1). TWICE: the projection of 2 v.
template <int K, int N, int ACC = 0, bool TWICE = false, class R>
__device__ __forceinline__ void project_pencil(const R (&v)[K + 1], R (&o)[N]) {
  constexpr int H = (K + 1) / 2;
  R s[H], d[H];
#pragma unroll
  for (int h = 0; h < H; ++h) {
    s[h] = v[K - h] + v[h];
    d[h] = v[K - h] - v[h];
  }
  auto p = [](int h, int n) { return TWICE ? pencil_tab<R, K>.P2[h][n] : pencil_tab<R, K>.P[h][n]; };
#pragma unroll
  for (int n = 0; n < N; ++n) {
    R acc = ACC ? o[n] : R(0);
    if (K % 2 == 0 && n % 2 == 0) acc = ACC ? acc - p(K / 2, n) * v[K / 2] : p(K / 2, n) * v[K / 2];
#pragma unroll
    for (int h = 0; h < H; ++h) {
      const R x = n % 2 ? d[h] : s[h];
      if (ACC) acc -= p(h, n) * x;
      else if (h == 0 && (K % 2 == 1 || n % 2 == 1)) acc = p(h, n) * x;
      else acc += p(h, n) * x;
    }
    o[n] = acc;
  }
}

// 2D transforms in registers: the triangle c[(b, x)], b + x <= n - 1, of 2D coefficients (ordered as the
// face modes) at the (K+1)^2 points, handed to put(q1, q2, value); and point values v[q1][q2] to the
// triangle o.
template <int K, int N, class R, class Put>
__device__ __forceinline__ void interp_triangle(const R (&c)[N * (N + 1) / 2], Put put) {
  R u[N][K + 1];  // [b][q2]
  static_for<N>([&](auto bc) {
    constexpr int B = decltype(bc)::value;
    R p[N - B];
#pragma unroll
    for (int x = 0; x < N - B; ++x) p[x] = c[tri(B + x) + x];
    interp_pencil<K, N - B>(p, u[B]);
  });
#pragma unroll
  for (int q2 = 0; q2 <= K; ++q2) {
    R p[N], v[K + 1];
#pragma unroll
    for (int b = 0; b < N; ++b) p[b] = u[b][q2];
    interp_pencil<K, N>(p, v);
#pragma unroll
    for (int q1 = 0; q1 <= K; ++q1) put(q1, q2, v[q1]);
  }
}
template <int K, int N, int ACC = 0, class R, class Get>
__device__ __forceinline__ void project_triangle(Get get, R (&o)[N * (N + 1) / 2]) {
  R u[N][K + 1];  // [b][q2]
#pragma unroll
  for (int q2 = 0; q2 <= K; ++q2) {
    R v[K + 1], p[N];
#pragma unroll
    for (int q1 = 0; q1 <= K; ++q1) v[q1] = get(q1, q2);
    project_pencil<K, N>(v, p);
#pragma unroll
    for (int b = 0; b < N; ++b) u[b][q2] = p[b];
  }
  static_for<N>([&](auto bc) {
    constexpr int B = decltype(bc)::value;
    R p[N - B];
#pragma unroll
    for (int x = 0; x < N - B; ++x) p[x] = ACC ? o[tri(B + x) + x] : R(0);
    project_pencil<K, N - B, ACC>(u[B], p);
#pragma unroll
    for (int x = 0; x < N - B; ++x) o[tri(B + x) + x] = p[x];
  });
}

// The warps of a CTA over the items of a phase. The items come in classes G = 0 .. NC-1 of
// count(G) items that take the same compile-time path (a pencil length); every class is cut into
// warp tasks of 32 items, and the tasks of all classes are dealt to the warps in turn.
template <int G, int NC, class Count, class F>
__device__ __forceinline__ void for_classes_(int t, int nw, int lane, Count count, F f) {
  if constexpr (G < NC) {
    constexpr int items = count(std::integral_constant<int, G>{});
    constexpr int tasks = (items + 31) / 32;
    for (; t < tasks; t += nw) {
      const int it = t * 32 + lane;
      if (items % 32 == 0 || it < items) f(std::integral_constant<int, G>{}, it);
    }
    for_classes_<G + 1, NC>(t - tasks, nw, lane, count, f);
  }
}
template <int NC, class Count, class F>
__device__ __forceinline__ void for_classes(int vw, int nw, int lane, Count count, F f) {
  for_classes_<0, NC>(vw, nw, lane, count, f);
}

__device__ __forceinline__ bool finite_bits(double x) { return (__double2hiint(x) & 0x7ff00000) != 0x7ff00000; }
__device__ __forceinline__ bool finite_bits(float x) { return (__float_as_int(x) & 0x7f800000) != 0x7f800000; }

}  // namespace dg
