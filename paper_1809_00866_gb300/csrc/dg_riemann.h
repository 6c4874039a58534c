// Exact Riemann solver of the artificial-compressibility system along a face normal (Sec. 2.1;
// device code of the face pass's residual modes).
//
// Works in units of the artificial speed: u = u_n / c, p / c^2. The 1-wave joins the left state to
// the star state, the 3-wave the right one; the 3-wave is the 1-wave of the mirrored problem
// (u -> -u), so one set of formulas serves both. Through (v, q) at star velocity u:
//   rarefaction (u >= v): p = q - 1/2 [u w(u) - v w(v) + asinh u - asinh v], w(x) = x + sqrt(x^2+1);
//   shock (u < v): p = q + (u - v)/s with the negative root s of s^2 - (v + u) s - 1 = 0, whose
//     inverse is -(S + Q)/2 with S = u + v, Q = sqrt(S^2 + 4): no division.
// The difference of the two asinh is asinh(u a(v) - v a(u)), a(x) = sqrt(x^2+1): an odd series in a
// small argument for the jumps of a resolved flow, where one asinh of u per iterate (about 70 FP64
// instructions) was half of the solver's time.
//
// Bound: the FP64 pipe. The star velocity is therefore found in FP32 first (safeguarded Newton, to
// about 1e-6), then corrected in FP64 by the cubic iteration of Chebyshev, u - d (1 + d phi''/(2 phi')),
// d = phi/phi', until |d| <= 3e-6: the error left is C3 |d|^3 with C3 = |phi''^2/(2 phi'^2) -
// phi'''/(6 phi')| at the root, below 2 over shocks and rarefactions alike, so below 6e-17 c. One
// FP64 evaluation usually does, and a last one at the star state gives the flux and its Jacobian. The residual's
// face pass at 13 x 9 x 11 P3: 512 -> 53 us against safeguarded Newton in FP64 throughout with two asinh per iterate.
#pragma once

namespace dg {

constexpr double kCubicStep = 3e-6;  // |phi/phi'| / c at which the FP64 iteration ends
constexpr int kCoarseIts = 8;        // FP32 iterations at most

// asinh(z)
__device__ __forceinline__ double asinh_jump(double z) {
  if (fabs(z) <= 0.125) {  // Taylor series; the first term left out is below 6e-19 |z|
    const double y = z * z;
    double s = 6435.0 / 557056.0;
    s = s * y - 143.0 / 10240.0;
    s = s * y + 231.0 / 13312.0;
    s = s * y - 63.0 / 2816.0;
    s = s * y + 35.0 / 1152.0;
    s = s * y - 5.0 / 112.0;
    s = s * y + 3.0 / 40.0;
    s = s * y - 1.0 / 6.0;
    return z + z * y * s;
  }
  return asinh(z);
}

struct AcWave {
  double p, d, dv, d2;  // p - q and its derivatives in u, v and twice in u
  double x, kap, iq;    // shock: (u - v)/Q, S/Q, 1/Q
};
// the 1-wave through (v, 0) at star velocity u; a = a(u), ia = 1/a, av = a(v)
__device__ __forceinline__ AcWave ac_wave(double u, double a, double ia, double v, double av) {
  AcWave r;
  if (u < v) {
    const double S = u + v, q2 = S * S + 4.0;
    r.iq = rsqrt(q2);
    const double Q = q2 * r.iq, du = u - v, is = -0.5 * (S + Q);
    r.x = du * r.iq;
    r.kap = S * r.iq;
    r.p = du * is;
    r.d = is * r.x + is;
    r.dv = is * r.x - is;
    r.d2 = is * r.iq * (2.0 + r.x - r.x * r.kap);
  } else {
    const double w = u + a, wv = v + av;
    r.p = -0.5 * (u * w - v * wv + asinh_jump(u * av - v * a));
    r.d = -w;
    r.dv = wv;
    r.d2 = -w * ia;
    r.x = r.kap = r.iq = 0.0;
  }
  return r;
}
// p and dp/du of the same in FP32
__device__ __forceinline__ void ac_wave_f(float u, float a, float v, float av, float& p, float& d) {
  if (u < v) {
    const float S = u + v, iq = rsqrtf(S * S + 4.0f), du = u - v, is = -0.5f * (S + (S * S + 4.0f) * iq);
    p = du * is;
    d = is + p * iq;
  } else {
    const float w = u >= 0.0f ? u + a : 1.0f / (a - u), wv = v >= 0.0f ? v + av : 1.0f / (av - v);
    p = -0.5f * (u * w - v * wv + __logf(w / wv));
    d = -w;
  }
}

// Star velocity to about 1e-6 (1 + |u|) in FP32, at most max_its iterations; adds their number to its.
__device__ __forceinline__ float ac_star_f(float ul, float ur, float dp, int max_its, int& its) {
  const float al = sqrtf(ul * ul + 1.0f), ar = sqrtf(ur * ur + 1.0f);
  const float scale = fabsf(ul) + fabsf(ur) + 1.0f;
  // two-rarefaction linearisation as the initial guess
  float u = (dp + ul * (ul + al) + ur * (ar - ur)) / ((ul + al) + (ar - ur));
  float lo = -1e30f, hi = 1e30f;
  for (int k = 0; k < max_its; ++k) {
    const float a = sqrtf(u * u + 1.0f);
    float p1, d1, p3, d3;
    ac_wave_f(u, a, ul, al, p1, d1);
    ac_wave_f(-u, a, -ur, ar, p3, d3);
    const float phi = dp + p1 - p3;
    if (phi > 0.0f) lo = u; else hi = u;
    float nxt = u - phi / (d1 + d3);
    if (!(nxt > lo && nxt < hi)) nxt = (lo > -1e29f && hi < 1e29f) ? 0.5f * (lo + hi) : nxt;
    const float step = nxt - u;
    u = nxt;
    ++its;
    if (fabsf(step) <= 1e-4f * scale) break;  // quadratic from here on
  }
  return u;
}

// Tangential-velocity ratio u_t(star)/u_t(v) across the 1-wave and its derivatives in u and v.
// Rarefaction: u_t w(u) invariant, w(x) = x + a = 1/(a - x), each w from the form whose terms have one sign
// (the other loses (u/c)^2 units of roundoff to cancellation; u is positive, or zero up to the band of a
// tie, where the side's ratio is used); shock: s [u_t] = [u_n u_t].
__device__ __forceinline__ void ac_tangential(const AcWave& k, double u, double a, double ia, double v, double av,
                                              double iav, double& t, double& tu, double& tv) {
  const bool shock = u < v;
  const double w = u + a, m = av + fabs(v);  // w(v), or its inverse where v < 0
  const double r = 1.0 / (shock ? 1.0 + k.x : (v >= 0.0 ? w : m * w));
  t = (shock ? 1.0 - k.x : (v >= 0.0 ? m : 1.0)) * r;
  if (shock) {
    const double f = 2.0 * k.iq * r * r;
    tu = f * (k.kap * k.x - 1.0);
    tv = f * (k.kap * k.x + 1.0);
  } else {
    tu = -t * ia;
    tv = t * iav;
  }
}

// Exact interface flux of the artificial-compressibility Riemann problem along the face
// normal, in the face's frame (n, t1, t2): inputs the normal and the two tangential velocity
// components and the pressure of each side, outputs F = (n.(u(x)u + pI) along n, t1, t2; u_n*)
// at the interface state, which is the star state, since the two acoustic waves always travel
// in opposite directions. The tangential velocity is taken from the side the contact (speed
// u*) comes from, the two sides averaged when |u*| is within a rounding band of zero. With
// J != nullptr also the flux's linearisation, 16 values from which the 4 x 8 Jacobian follows
// (its other entries are zero or multiples of these): with du* = J0 . (un_L, p_L, un_R, p_R),
//   dF_n = J1 . (un_L, p_L, un_R, p_R),   dF_p = du*,
//   dF_t = A_t du* + B_t dun_L + C_t dun_R + D dt_L + E dt_R   (t = t1, t2),
// stored J0[4], J1[4], A_1, A_2, D, E, B_1, C_1, B_2, C_2.
__device__ __forceinline__ void ac_riemann(double unl, double t1l, double t2l, double pL, double unr, double t1r,
                                           double t2r, double pR, double c, double (&F)[4], double* J,
                                           unsigned* status, int max_its) {
  const double ic = 1.0 / c, c2 = c * c;
  const double ul = unl * ic, ur = unr * ic, dp = (pL - pR) * (ic * ic);
  const double al2 = ul * ul + 1.0, ar2 = ur * ur + 1.0;
  const double ial = rsqrt(al2), iar = rsqrt(ar2), al = al2 * ial, ar = ar2 * iar;
  const double scale = fabs(ul) + fabs(ur) + 1.0;
  int it = 0;
  double us = (double)ac_star_f((float)ul, (float)ur, (float)dp, max_its < kCoarseIts ? max_its : kCoarseIts, it);
  if (!(fabs(us) < 1e30)) us = (dp + ul * (ul + al) + ur * (ar - ur)) / ((ul + al) + (ar - ur));  // beyond FP32
  double lo = -1e300, hi = 1e300;
  bool ok = false;
  for (; it < max_its; ++it) {
    const double a2 = us * us + 1.0, ia = rsqrt(a2), a = a2 * ia;
    const AcWave k1 = ac_wave(us, a, ia, ul, al), k3 = ac_wave(-us, a, ia, -ur, ar);
    const double phi = dp + k1.p - k3.p, r = 1.0 / (k1.d + k3.d);  // 1 / phi', < 0
    if (phi > 0.0) lo = us; else hi = us;
    const double d = phi * r;
    double nxt = us - d * (1.0 + 0.5 * d * (k1.d2 - k3.d2) * r);
    if (!(nxt > lo && nxt < hi)) nxt = us - d;
    const bool in = nxt > lo && nxt < hi;
    if (!in) nxt = (lo > -1e299 && hi < 1e299) ? 0.5 * (lo + hi) : nxt;
    const double step = nxt - us;
    us = nxt;
    if (fabs(step) <= 1e-15 * scale || (in && fabs(d) <= kCubicStep)) { ok = true; break; }
  }
  if (!ok && status) atomicOr(status, (unsigned)DG_STATUS_RIEMANN);
  const double a2 = us * us + 1.0, ia = rsqrt(a2), a = a2 * ia;
  const AcWave k1 = ac_wave(us, a, ia, ul, al), k3 = ac_wave(-us, a, ia, -ur, ar);
  const double band = 1e-12 * scale;
  const bool tie = us >= -band && us <= band;
  // weighted ratios of the left and right side and their derivatives: one evaluation for the side that the contact
  // comes from, whichever it is in a lane (one per side took every warp through both), a second in a tie
  double tl = 0.0, tlu = 0.0, tlv = 0.0, tr = 0.0, tru = 0.0, trv = 0.0;
  auto side = [&](bool left, double weight) {
    double t, tu, tv;
    AcWave k;
    k.x = left ? k1.x : k3.x;
    k.kap = left ? k1.kap : k3.kap;
    k.iq = left ? k1.iq : k3.iq;
    ac_tangential(k, left ? us : -us, a, ia, left ? ul : -ur, left ? al : ar, left ? ial : iar, t, tu, tv);
    if (left) {
      tl = weight * t; tlu = weight * tu; tlv = weight * tv;
    } else {
      tr = weight * t; tru = -weight * tu; trv = -weight * tv;
    }
  };
  const bool left = us > 0.0;
  side(left, tie ? 0.5 : 1.0);
  if (tie) side(!left, 0.5);
  F[0] = c2 * (us * us + k1.p) + pL;
  F[3] = c * us;
  const double T1 = tl * t1l + tr * t1r, T2 = tl * t2l + tr * t2r;
  F[1] = F[3] * T1;
  F[2] = F[3] * T2;
  if (J) {
    // implicit-function derivatives of u* and p* with respect to (ul, pl, ur, pr), in units of c
    const double r = 1.0 / (k1.d + k3.d);
    const double u_l = -k1.dv * r, u_r = -k3.dv * r;  // d u* / d ul, d u* / d ur
    const double q = 2.0 * us + k1.d;                 // dF_n = q du* + dv_1 dul + dpl
    J[0] = u_l;
    J[1] = -r * ic;
    J[2] = u_r;
    J[3] = r * ic;
    J[4] = c * (q * u_l + k1.dv);
    J[5] = 1.0 - q * r;
    J[6] = c * (q * u_r);
    J[7] = q * r;
    J[8] = us * (tlu * t1l + tru * t1r) + T1;
    J[9] = us * (tlu * t2l + tru * t2r) + T2;
    J[10] = F[3] * tl;
    J[11] = F[3] * tr;
    J[12] = us * tlv * t1l;
    J[13] = us * trv * t1r;
    J[14] = us * tlv * t2l;
    J[15] = us * trv * t2r;
  }
}

}  // namespace dg
