"""Host build of the FP64 reciprocals and roots that start in single precision
(paper_2503_12557_gb300/csrc/peps_newton.cuh, plain scalar code), against long double: what the QR's
reflectors and the cutoff eigendecomposition's rotations are formed from is as accurate as with sqrt and
division.

Bounds: the last sum rounds once, 0.5 ulp; the residual 1 - (x r) and x - s s are exact up to 2^-40 of an
ulp (one rounding of a fused product), but 1 - (x y) y has the rounding of x y in it, which enters halved: up
to 0.5 ulp more.  So 0.52 for the reciprocal and the root and 1.02 for the reciprocal root, with a
single-precision start two units off.  A reflector's scalars (tau, 1 / (alpha - beta)) and a rotation's cosine
may not be further off than by sqrt and divisions on the same arguments (a final rounding allowed for).
"""
import os
import shutil
import subprocess

import pytest

HDR = os.path.join(os.path.dirname(__file__), "..", "paper_2503_12557_gb300", "csrc")

DRIVER = r"""
#define __device__
#define __forceinline__ inline
#include <cmath>
#include <cstdio>
#include <cstring>
#include <random>
static std::mt19937_64 g(1);
static float off(float x) { int b; memcpy(&b, &x, 4); b += (int)(g() % 5) - 2; memcpy(&x, &b, 4); return x; }
static float rsqrtf(float x) { return off((float)(1.0 / sqrt((double)x))); }
static float __frcp_rn(float x) { return 1.0f / x; }
using std::fma;
#include "peps_newton.cuh"
using namespace peps;
typedef long double ld;
static double err(double v, ld e) { return fabs((double)((ld)v - e)) / ldexp(1.0, ilogb((double)e) - 52); }
int main() {
  double w[10] = {0};
  auto up = [&](int i, double v, ld e) { const double d = err(v, e); if (d > w[i]) w[i] = d; };
  std::uniform_real_distribution<double> U(-1, 1);
  for (int k = 0; k < 2000000; ++k) {
    const double x = pow(10, 15 * U(g));
    up(0, rsqrt_nr(x), 1 / sqrtl((ld)x));
    up(1, rcp_nr(x), 1 / (ld)x);
    up(2, sqrt_nr(x, rsqrt_nr(x)), sqrtl((ld)x));
    // a reflector of a column with head a and squared tail norm s
    const double a = U(g) * pow(10, 3 * U(g)), s = pow(10, 6 * U(g)), n2 = fma(a, a, s), y = rsqrt_nr(n2);
    const double nrm = sqrt_nr(n2, y), o = sqrt(a * a + s), ob = a >= 0 ? -o : o;
    const ld ne = sqrtl((ld)a * a + s);
    up(3, fma(fabs(a), y, 1.0), 1 + fabsl((ld)a) / ne);
    up(4, (ob - a) / ob, 1 + fabsl((ld)a) / ne);
    up(5, rcp_nr(fabs(a) + nrm), 1 / (fabsl((ld)a) + ne));
    up(6, fabs(1.0 / (a - ob)), 1 / (fabsl((ld)a) + ne));
    // the cosine of a Jacobi rotation with difference d and off-diagonal entry x / 2
    const double d = U(g) * pow(10, 3 * U(g)), q = U(g) * pow(10, 3 * U(g)), h2 = fma(d, d, q * q);
    const double t = (d < 0 ? -q : q) * rcp_nr(fabs(d) + h2 * rsqrt_nr(h2));
    const ld te = (d < 0 ? -(ld)q : (ld)q) / (fabsl((ld)d) + sqrtl((ld)d * d + (ld)q * q));
    const double ta = d / q, to = copysign(1.0, ta) / (fabs(ta) + sqrt(1.0 + ta * ta));
    up(7, rsqrt_nr(fma(t, t, 1.0)), 1 / sqrtl(1 + te * te));
    up(8, 1.0 / sqrt(1.0 + to * to), 1 / sqrtl(1 + te * te));
  }
  for (int i = 0; i < 9; ++i) printf("%.4f ", w[i]);
  return 0;
}
"""


def test_single_precision_starts(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    src, exe = tmp_path / "drv.cpp", tmp_path / "drv"
    src.write_text(DRIVER)
    subprocess.run([cxx, "-O2", "-std=c++17", "-ffp-contract=off", "-I", os.path.abspath(HDR), str(src), "-o", str(exe)],
                   check=True, capture_output=True)
    w = [float(v) for v in subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split()]
    assert w[0] <= 1.02 and max(w[1:3]) <= 0.52
    assert w[3] <= w[4] and w[5] <= w[6] + 0.52 and w[7] <= w[8] + 0.52
