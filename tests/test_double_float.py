"""Double-float arithmetic of the mixed mode under any contraction (no GPU needed).

The header is compiled for the host with a number type in place of float that
contracts wherever a compiler may: a product keeps its unrounded value, and an
addition takes that one, as a fused multiply-add would.  Only the named
intrinsics round by themselves.  Against exact values, the results must keep the
accuracy the header states (a few 2^-46): 2^-44 of the sum of the terms'
magnitudes for products, sums and invariants, 2^-43 for quotients and roots,
which take a product more.
"""
import os
import shutil
import subprocess

import pytest

from paper_2106_12631_gb300 import build as B

SRC = r'''
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstdlib>
typedef float real32;
struct cfl {  // a float whose last operation, if a product, is still open to contraction
  real32 v;
  double exact;
  bool open;
  cfl() = default;
  cfl(real32 x) : v(x), exact(x), open(false) {}
  explicit cfl(double x) : v((real32)x), exact(v), open(false) {}
  explicit operator double() const { return v; }
};
static cfl operator*(cfl a, cfl b) {
  cfl r((real32)(a.v * b.v));
  r.exact = (double)a.v * b.v;
  r.open = true;
  return r;
}
static cfl operator-(cfl a) { a.v = -a.v; a.exact = -a.exact; return a; }
static cfl operator+(cfl a, cfl b) { return cfl(a.open ? a.exact + (double)b.v : (double)a.v + (b.open ? b.exact : (double)b.v)); }
static cfl operator-(cfl a, cfl b) { return a + (-b); }
static cfl operator/(cfl a, cfl b) { return cfl((real32)(a.v / b.v)); }
static bool operator<(cfl a, cfl b) { return a.v < b.v; }
static cfl fmaf(cfl a, cfl b, cfl c) { return cfl((real32)std::fma(a.v, b.v, c.v)); }
static cfl fmac(cfl a, cfl b, cfl c) { return fmaf(a, b, c); }
static cfl fabsf(cfl a) { a.v = std::fabs(a.v); a.exact = std::fabs(a.exact); return a; }
static cfl rsqrtf(cfl a) { return cfl((real32)(1.0 / std::sqrt((double)a.v))); }
static cfl __fmul_rn(cfl a, cfl b) { return cfl((real32)(a.v * b.v)); }
static cfl __fadd_rn(cfl a, cfl b) { return cfl((real32)(a.v + b.v)); }
#define __device__
#define __forceinline__ inline
#define float cfl
#include "dfl.cuh"
#undef float
using namespace mg;
static double unit() { return (std::rand() + 0.5) / (RAND_MAX + 1.0) * 2 - 1; }
static long double val(dfl a) { return (long double)a.hi.v + a.lo.v; }
int main() {
  double sum = 0, inv = 0, quo = 0;
  for (int n = 0; n < 200000; ++n) {
    const double s = std::ldexp(1.0, std::rand() % 12);
    const dfl a = dfl_split(s * unit()), b = dfl_split(unit()), c = dfl_split(unit()), d = dfl_split(s * unit());
    const long double ab = val(a) * val(b), cd = val(c) * val(d);
    const dfl r = dfl_add(dfl_mul(a, b), dfl_mul(c, d));
    sum = std::fmax(sum, (double)(std::fabs(val(r) - (ab + cd)) / (std::fabs(ab) + std::fabs(cd))));
    const dfl t = dfl_add(dfl_mul(a, a), dfl_mul(b, b));
    const long double x = val(a) * val(a) + val(b) * val(b);
    quo = std::fmax(quo, (double)std::fabs(val(dfl_rsqrt(t)) * std::sqrt(x) - 1));
    quo = std::fmax(quo, (double)std::fabs(val(dfl_rcp(t)) * x - 1));
    // a sum of two nearly light-like momenta: large squares that cancel
    double k[4] = {0, 0, 0, 0};
    for (int i = 0; i < 2; ++i) {
      double p[3] = {s * unit(), s * unit(), s * unit()};
      k[0] += std::sqrt(p[0] * p[0] + p[1] * p[1] + p[2] * p[2]);
      for (int j = 0; j < 3; ++j) k[j + 1] += p[j];
    }
    DflSum<cfl> q[4];
    long double k2 = 0, mag = 0;
    for (int mu = 0; mu < 4; ++mu) {
      const dfl h = dfl_split(k[mu]);
      q[mu].first(h.hi, h.lo);
      k2 += (mu == 0 ? 1 : -1) * val(h) * val(h);
      mag += val(h) * val(h);
    }
    const DflSum<cfl> m = dfl_invariant(q);
    inv = std::fmax(inv, (double)(std::fabs((long double)m.s.v + m.err.v - k2) / mag));
  }
  std::printf("%.17g %.17g %.17g\n", sum, inv, quo);
}
'''


@pytest.mark.skipif(shutil.which("g++") is None, reason="g++ not available")
def test_accuracy_does_not_depend_on_contraction(tmp_path):
    src, exe = tmp_path / "probe.cpp", tmp_path / "probe"
    src.write_text(SRC)
    r = subprocess.run(["g++", "-std=c++17", "-O1", "-ffp-contract=off", "-w", "-I", B.CSRC, str(src), "-o", str(exe)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
    out = subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout
    err_sum, err_inv, err_quo = (float(x) for x in out.split())
    assert err_sum <= 2.0 ** -44 and err_inv <= 2.0 ** -44 and err_quo <= 2.0 ** -43, out
