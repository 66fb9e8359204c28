"""The fixed-point arithmetic of csrc/fdlbm_fx.cuh, compiled for the host, against 113-bit floating point.

A bracket n F_k E or n F_k O is a sum of two products and, for E, a constant, in units of 2^ex. In units of
the last place: a ring constant carries 1 (2 of its product, shifted down by 2 or more), a power of p 2
(X = p^2 within 2, X^2 and A1 X within 6, two bits down), each product drops 2; so two products and A0
(1.5) stay within 2 (1/4 + 2 + 2) + 1.5 = 10, |q| being at most 1/4 and |c| at most 1. The form with one
scale for all rings (FP32 storage) takes its powers at ring 4's scale, without the two bits: 2 (1 + 6 + 2)
+ 4 = 22 units. Rounding must have no sign either, since a bias of f adds up over a solve: the mean over
N nodes of errors below 1 unit rms stays within 5 / sqrt(N) of what is left, 1/16 unit.
"""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(__file__), "..", "paper_0801_4169_gb300", "csrc")
SRC = r"""
#define __host__
#define __device__
#define __forceinline__ inline
#include "fdlbm_fx.cuh"
using namespace fdlbm::fx;
#if __LDBL_MANT_DIG__ >= 113
typedef long double quad;
#else
typedef __float128 quad;
#endif
static const int VS[4] = {100, 192, 299, 449};
static s64 frac(int V, int power, unsigned long long den, int e) {
  unsigned __int128 n = 1;
  for (int i = 0; i < power; ++i) n *= V;
  return (s64)(((n << (62 - e)) + den / 2) / den);
}
// Errors of the pairs of n nodes, in units of 2^ex: out[node][ring][direction][E, O].
extern "C" int pairs(int plain, int n, const double* ux, const double* uy, const double* T, const double* nF,
                     double* out) {
  const double s = 0.70710678118654752440;
  int bad = 0;
  for (int i = 0; i < n; ++i) {
    const double px = ux[i] / T[i], py = uy[i] / T[i], p[4] = {px, s * (px + py), py, s * (py - px)};
    const double b2 = ux[i] * px + uy[i] * py, A1 = 1 - 0.5 * b2, A0 = A1 + 0.125 * b2 * b2;
    const Base b = base_of(A0, A1, p[0], p[1], p[2], p[3]);
    if (!b.ok) { ++bad; continue; }
    for (int k = 0; k < 4; ++k) {
      const int own = plain ? k : 3, es = scale_of(b, own);
      const s64 c[4] = {frac(VS[k], 2, 20000, exp_c1(own)), frac(VS[k], 4, 2400000000ull, exp_c2(own)),
                        frac(VS[k], 1, 100, exp_c3(own)), frac(VS[k], 3, 6000000, exp_c4(own))};
      const double w = nF[4 * i + k];
      const RingFx r = plain ? ring_scaled(b.A0f, es, b.e0, b.ea, b.ep, k, w, c)
                             : ring_shared(limb(b.A0f >> imin(es - b.e0, 63)), es, w, c);
      const quad v = (quad)VS[k] / 100, u = std::ldexp(1.0, r.ex);
      for (int t = 0; t < 4; ++t) {
        const Powers pw = powers_of(b, p[t], plain ? 2 : 0);
        s64 E, O;
        if (plain) pair_of<true>(r, dir_plain(pw), E, O);
        else pair_of<false>(r, dir_shared(pw, b, es), E, O);
        const quad P = p[t] < 0 ? -p[t] : p[t];
        const quad ee = (quad)w * ((quad)A0 + v * v / 2 * (quad)A1 * P * P + v * v * v * v / 24 * P * P * P * P);
        const quad oo = (quad)w * (v * (quad)A1 * P + v * v * v / 6 * P * P * P);
        out[((4 * i + k) * 4 + t) * 2] = (double)((quad)E - ee / u);
        out[((4 * i + k) * 4 + t) * 2 + 1] = (double)((quad)O - oo / u);
        const quad lim = (s64)1 << 60;
        if ((quad)E > lim || -(quad)E > lim || (quad)O > lim || -(quad)O > lim) ++bad;
      }
    }
  }
  return bad;
}
extern "C" void conv(int n, const long long* R, const int* ex, double* nearest, double* fast) {
  for (int i = 0; i < n; ++i) nearest[i] = to_f64(R[i], ex[i]), fast[i] = to_f64_fast(R[i], ex[i]);
}
"""


@pytest.fixture(scope="module")
def fx(tmp_path_factory):
    if not shutil.which("g++"):
        pytest.skip("no g++")
    d = tmp_path_factory.mktemp("fx")
    src = d / "fx.cc"
    src.write_text(SRC)
    subprocess.run(["g++", "-O2", "-shared", "-fPIC", "-ffp-contract=off", "-I", CSRC, "-o", str(d / "fx.so"), str(src)],
                   check=True)
    return ctypes.CDLL(str(d / "fx.so"))


def _p(a):
    return a.ctypes.data_as(ctypes.c_void_p)


# (|u|, theta): at rest, ordinary, hypersonic (b = u^2 / 2 theta up to 60), nearly cold, large numbers
@pytest.mark.parametrize("u,T", [(0.0, 1.0), (1e-9, 1.0), (0.7, 1.0), (8.42, 175.8), (19.6, 76.8), (11.0, 1.0),
                                 (0.3, 4e-3), (300.0, 9000.0)])
@pytest.mark.parametrize("plain", [1, 0])
def test_pairs_within_their_units_and_without_bias(fx, plain, u, T):
    rng = np.random.default_rng(7)
    n = 4000
    a = rng.uniform(0, 2 * np.pi, n)
    if u == 8.42:
        a[:] = 0.0  # a projection of exactly zero
    uu = u * (1 + 1e-3 * rng.standard_normal(n))
    ux, uy = uu * np.cos(a), uu * np.sin(a)
    th = T * (1 + 1e-3 * rng.standard_normal(n))
    nF = rng.standard_normal((n, 4)) * 10.0 ** rng.uniform(-6, 6, (n, 4))
    out = np.zeros((n, 4, 4, 2))
    assert fx.pairs(plain, n, _p(ux), _p(uy), _p(th), _p(nF), _p(out)) == 0
    assert np.abs(out).max() <= (10.0 if plain else 22.0)
    if plain:
        assert np.abs(out.mean(axis=(0, 1, 2))).max() <= 1 / 16 + 5 / np.sqrt(n * 16)


def test_infinite_and_extreme_numbers_leave_the_fixed_point_range(fx):
    nF = np.ones((1, 4))
    out = np.zeros((1, 4, 4, 2))
    for ux, T in ((np.inf, 1.0), (np.nan, 1.0), (1.0, np.nan), (5000.0, 1.0), (2e9, 1.0)):
        x, y, t = np.array([ux]), np.zeros(1), np.array([T])
        with np.errstate(all="ignore"):
            assert fx.pairs(1, 1, _p(x), _p(y), _p(t), _p(nF), _p(out)) == 1


def test_integers_round_to_the_nearest_even_double(fx):
    rng = np.random.default_rng(1)
    bits = rng.integers(0, 63, 20000)
    R = (rng.integers(0, 2**62, 20000) >> bits) * rng.choice([-1, 1], 20000)
    tie = ((rng.integers(2**52, 2**53, 2000) << 8) | 128) * rng.choice([-1, 1], 2000)  # halfway cases
    edge = np.array([0, 1, -1, 2**31 - 1, 2**31, 2**32 - 1, 2**32, -(2**32), 2**53 - 1, 2**53 + 1, 2**62 - 1, 1 - 2**62])
    R = np.concatenate([R, tie, edge]).astype(np.int64)
    ex = rng.integers(-900, 900, R.size).astype(np.int32)
    a, b = np.zeros(R.size), np.zeros(R.size)
    fx.conv(R.size, _p(R), _p(ex), _p(a), _p(b))
    ref = np.array([float(int(r)) for r in R])  # Python rounds to nearest even
    assert np.array_equal(a, np.ldexp(ref, ex))
    big = np.abs(R) >= 2**32
    assert np.array_equal(b[big], np.ldexp(ref, ex)[big])
