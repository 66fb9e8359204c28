"""fx::from_f64_rn of csrc/fdlbm_fx.cuh, compiled for the host: FP64 to fixed point, to nearest even at every exponent, as
the viscosity enters the integer weights of Eq. 17."""
import ctypes
import os
import shutil
import subprocess
from fractions import Fraction

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(__file__), "..", "paper_0801_4169_gb300", "csrc")
SRC = r"""
#define __host__
#define __device__
#define __forceinline__ inline
#include "fdlbm_fx.cuh"
extern "C" void conv(int n, const double* x, const int* e, long long* out) {
  for (int i = 0; i < n; ++i) out[i] = fdlbm::fx::from_f64_rn(x[i], e[i]);
}
"""


def test_fixed_point_numbers_round_to_nearest_even(tmp_path):
    if not shutil.which("g++"):
        pytest.skip("no g++")
    src, lib = tmp_path / "r.cc", tmp_path / "r.so"
    src.write_text(SRC)
    subprocess.run(["g++", "-O2", "-shared", "-fPIC", "-I", CSRC, "-o", str(lib), str(src)], check=True)
    rng = np.random.default_rng(3)
    e = rng.integers(3, 8, 20000).astype(np.int32)  # units of 2^-59 to 2^-55
    x = rng.uniform(0.5, 1.0, e.size) * 2.0 ** -rng.integers(0, 70, e.size) * rng.choice([-1.0, 1.0], e.size)
    ties = (rng.integers(1, 2**40, 2000) + 0.5) * 2.0 ** (e[:2000] - 62.0)
    x[:2000] = ties * rng.choice([-1.0, 1.0], 2000)
    x[2000:2004] = [0.0, -0.0, 2.0**-62, 0.5]
    out = np.zeros(x.size, dtype=np.int64)
    p = lambda a: a.ctypes.data_as(ctypes.c_void_p)  # noqa: E731
    ctypes.CDLL(str(lib)).conv(x.size, p(x), p(e), p(out))
    # Python rounds a fraction to the nearest integer, ties to even
    assert [int(o) for o in out] == [round(Fraction(float(a)) * 2 ** int(62 - k)) for a, k in zip(x, e)]
