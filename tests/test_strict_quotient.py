"""The quotient of FDLBM_FP64_STRICT's equilibrium (csrc/fdlbm_strict.cu, dvd_by): two correction steps from the
correctly rounded reciprocal give the correctly rounded quotient, here on the host against IEEE division, with
significands drawn at random, all ones, almost all ones and with few bits set."""
import ctypes
import shutil
import subprocess

import pytest

SRC = r"""
#include <math.h>
#include <stdint.h>
#include <string.h>
static uint64_t s = 88172645463325252ull;
static uint64_t next(void) { s ^= s << 13; s ^= s >> 7; s ^= s << 17; return s; }
static double number(int kind, int span) {
  uint64_t m = next() & 0xfffffffffffffull;
  if (kind == 1) m = 0xfffffffffffffull;
  if (kind == 2) m |= 0xffffffffff000ull;
  if (kind == 3) m &= 0xfff0000000000ull;
  if (kind == 4) m &= 0xfffull;
  const uint64_t u = m | (uint64_t)(1023 - span + (int)(next() % (2 * span))) << 52;
  double x;
  memcpy(&x, &u, 8);
  return x;
}
long mismatches(long n) {
  long bad = 0;
  for (long i = 0; i < n; ++i) {
    const double a = number((int)(i % 5), 590), b = number((int)(i / 5 % 5), 205), y = 1.0 / b;
    const double q0 = a * y, q1 = fma(fma(-b, q0, a), y, q0);
    bad += fma(fma(-b, q1, a), y, q1) != a / b;
  }
  return bad;
}
"""


def test_two_corrections_give_the_rounded_quotient(tmp_path):
    if not shutil.which("gcc"):
        pytest.skip("no gcc")
    src, lib = tmp_path / "q.c", tmp_path / "q.so"
    src.write_text(SRC)
    subprocess.run(["gcc", "-O2", "-shared", "-fPIC", "-ffp-contract=off", "-o", str(lib), str(src), "-lm"], check=True)
    f = ctypes.CDLL(str(lib)).mismatches
    f.restype, f.argtypes = ctypes.c_long, [ctypes.c_long]
    assert f(3_000_000) == 0
