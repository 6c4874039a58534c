"""The tangential flux of the Riemann solver where the normal velocity is many times the artificial speed c.

Across a rarefaction u_t (u + a) is invariant, a = sqrt(u^2 + c^2) (Sec. 2.1), so that
u_t(star)/u_t(v) = (v + a(v)) / (u + a(u)). With w(x) = x + a(x) = c^2 / (a(x) - x) taken in the form whose
terms have one sign, every operand carries a few roundings: at most three for each w, one for the quotient,
the product or two around it, and two for the flux, ten units of 1.1e-16 in all; the bound is 4e-15. In the
other form the relative error grows as (u/c)^2.

The header is compiled for the host and compared in 40-digit arithmetic at the star velocity that it
returns itself. The kernels are compared with the oracle in a flow whose components are all positive: there
the oracle's ratios have terms of one sign too, and its shocks, which lose (u/c)^2 units of roundoff of
the velocity jump, are good to 2e-13 at |u|/c = 50; the bound is 1e-12 as in the other operator tests.
"""
import ctypes
import os
import subprocess

import numpy as np
import pytest

import oracle as O
import synthetic as S
from _gpu_common import dev, host, pair, rel

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1809_00866_gb300", "csrc")
SHIM = r"""
#include <cmath>
#define __device__
#define __forceinline__ inline
#define DG_STATUS_RIEMANN 1u
static inline double rsqrt(double x) { return 1.0 / std::sqrt(x); }
static inline float rsqrtf(float x) { return 1.0f / std::sqrt(x); }
static inline float host_logf(float x) { return std::log(x); }
#define __logf host_logf
static inline unsigned atomicOr(unsigned* p, unsigned v) { *p |= v; return 0; }
using std::asinh;
using std::fabs;
#include "dg_riemann.h"
extern "C" unsigned flux(const double* l, const double* r, double c, double* F, double* J) {
  unsigned status = 0;
  double f[4];
  dg::ac_riemann(l[0], l[1], l[2], l[3], r[0], r[1], r[2], r[3], c, f, J, &status, 60);
  for (int i = 0; i < 4; ++i) F[i] = f[i];
  return status;
}
"""


@pytest.fixture(scope="module")
def flux(tmp_path_factory):
    d = tmp_path_factory.mktemp("riemann")
    (d / "shim.cpp").write_text(SHIM)
    so = str(d / "shim.so")
    subprocess.check_call(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, "-o", so, str(d / "shim.cpp")])
    L = ctypes.CDLL(so)
    p = ctypes.POINTER(ctypes.c_double)
    L.flux.argtypes = [p, p, ctypes.c_double, p, p]

    def call(l, r, c):
        l, r, F, J = np.array(l, float), np.array(r, float), np.zeros(4), np.zeros(16)
        assert L.flux(*(a.ctypes.data_as(p) for a in (l, r)), c, *(a.ctypes.data_as(p) for a in (F, J))) == 0
        return F, J
    return call


@pytest.mark.parametrize("sign", [1, -1])
@pytest.mark.parametrize("R", [0.1, 1.0, 10.0, 100.0, 1000.0])
def test_rarefaction_ratio(flux, R, sign):
    mp = pytest.importorskip("mpmath")
    mp.mp.dps = 40
    rng = np.random.default_rng(int(70 * R) + sign)
    a = lambda x: mp.sqrt(x * x + 1)
    seen = {1: 0, -1: 0}
    for n in range(200):
        c = 0.25  # a power of two: the velocities in units of c are exact
        v = R * rng.uniform(0.5, 1.0) * (1 if n % 2 else -1)  # upwind side's normal velocity, towards the face or away
        dp = (1.0 if v > 0 else 30.0) * R * R * rng.uniform(0.5, 1.0)  # drives the star velocity above it
        o = v * 1.3 + 0.1
        up, dn = [sign * v * c, 1.0, 0.5, dp * c * c], [sign * o * c, 0.3, -0.7, 0.0]
        F, J = flux(up, dn, c) if sign > 0 else flux(dn, up, c)
        u, w = mp.mpf(sign * F[3]) / c, mp.mpf(v)
        if u <= mp.mpf("1e-3") or u < w:
            continue  # a shock, or within reach of the tie band
        seen[1 if v > 0 else -1] += 1
        t = (w + a(w)) / (u + a(u))
        tt = F[3] * t  # dF_t / du_t of the upwind side
        for got, want in ((F[1], F[3] * t * up[1]), (F[2], F[3] * t * up[2]), (J[10 if sign > 0 else 11], tt),
                          (J[12 if sign > 0 else 13], F[3] / c * t * up[1] * sign / a(w)),
                          (J[14 if sign > 0 else 15], F[3] / c * t * up[2] * sign / a(w))):
            assert abs((got - want) / want) < 4e-15
    assert seen[1] > 20 and (seen[-1] > 20 or R < 1.0)


@pytest.mark.gpu
@pytest.mark.parametrize("dims,k", [((2, 3, 3), 2), ((3, 4, 5), 3), ((3, 2, 3), 4)])
def test_fast_flow_matches_oracle(dims, k):
    xs = [S.perturbed_nodes(n, seed=s) for n, s in zip(dims, (1, 2, 3))]
    dg, m = pair(*xs, [k], c=0.02)  # |u|/c = 50, 40 and 30 along the axes
    w = 0.1 * O.project_tgv(m) + S.perturbation(m.ne, k, 0.02, 4)
    vol = np.einsum("i,j,l->lji", *[np.diff(x) for x in xs]).reshape(-1)
    for i, u in enumerate((1.0, 0.8, 0.6)):
        w[:, i, 0] += u * np.sqrt(vol)  # the constant u: its coefficient is u sqrt(|K|)
    v = S.direction(m.ne, k, 5)
    out = dg.empty()
    dg.dg_residual(dev(w), out)
    assert rel(host(out), O.residual(m, w)) < 1e-12
    dg.dg_set_linearization(dev(w), 0.7)
    dg.dg_jvp(dev(v), out)
    assert rel(host(out), O.jvp(m, w, v, 0.7)) < 1e-12
    assert dg.dg_get_status() == 0
