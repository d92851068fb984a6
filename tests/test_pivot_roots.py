"""Reciprocals and reciprocal roots of pivots (csrc/feti_root.cuh), on the CPU.

The device functions are compiled by g++ with the intrinsics they use written
out: __frcp_rn is the rounded FP32 reciprocal, rsqrtf any FP32 number within two
ulps of the reciprocal root (its documented error).  Against long double over
all binary exponents of normal numbers.  Bounds: the truncated 24-bit mantissa
and the seed are off by e < 2^-21.5, the third-order step leaves e^3 < 2^-64 and
two roundings of the result's own size: 1 ulp for the reciprocal and the root
(2^-52).  Pivots from 2^1021 on are scaled by 2^-64 first (k_tcc_diag): their
reciprocal is not asked for.
"""
import subprocess

from fake_cuda import CSRC, cuda_include

PROGRAM = r"""
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <random>
#define __device__
#define __forceinline__ inline
#include <algorithm>
using std::max; using std::min; using std::fma; using std::isfinite;
static std::mt19937_64 gen(7);
static int64_t bits(double x) { int64_t v; memcpy(&v, &x, 8); return v; }
static int __double2hiint(double x) { return (int)(bits(x) >> 32); }
static int __double2loint(double x) { return (int)bits(x); }
static long long __double_as_longlong(double x) { return bits(x); }
static double __hiloint2double(int hi, int lo) {
  const uint64_t v = (uint64_t)(uint32_t)hi << 32 | (uint32_t)lo;
  double x; memcpy(&x, &v, 8); return x;
}
static float __int_as_float(int v) { float x; memcpy(&x, &v, 4); return x; }
static int __float_as_int(float x) { int v; memcpy(&v, &x, 4); return v; }
static float __frcp_rn(float x) { return 1.0f / x; }
static float seed_root(float x) {
  return __int_as_float(__float_as_int((float)(1.0L / sqrtl((long double)x))) + (int)(gen() % 5) - 2);
}
#define rsqrtf seed_root
#define asm(...)
#include "feti_root.cuh"
#undef asm

static int wrong = 0;
static void check(const char* what, double got, long double exact, double d, double ulps) {
  const long double ulp = ldexpl(1.0L, std::max(ilogbl(exact), -1022) - 52);
  if (fabsl((long double)got - exact) <= ulps * ulp) return;
  if (wrong++ < 5) printf("%s of %a: %a, not %La\n", what, d, got, exact);
}
int main() {
  std::uniform_real_distribution<double> u(1.0, 2.0);
  for (int e = -1022; e <= 1023; ++e)
    for (int i = 0; i < 200; ++i) {
      const double m = i == 0 ? 1.0 : i == 1 ? std::nextafter(2.0, 0.0) : u(gen), d = std::ldexp(m, e);
      if (e < 1021) check("recip", feti::recip(d), 1.0L / d, d, 1.0);
      check("inv_sqrt", feti::inv_sqrt(d), 1.0L / sqrtl(d), d, 1.0);
      if (!feti::positive(d) || feti::positive(-d)) ++wrong;
    }
  for (double x : {0.0, -0.0, (double)INFINITY, -(double)INFINITY, (double)NAN})
    if (feti::positive(x)) ++wrong;
  return wrong ? 1 : 0;
}
"""


def test_against_long_double(tmp_path):
    src = tmp_path / "roots.cpp"
    src.write_text(PROGRAM)
    exe = str(tmp_path / "roots")
    subprocess.run(["g++", "-std=c++17", "-O1", "-ffp-contract=off", str(src), "-o", exe, "-I", CSRC,
                    "-I", cuda_include(), "-I", "/usr/local/cuda/include"], check=True)
    done = subprocess.run([exe], timeout=120, capture_output=True, text=True)
    assert done.returncode == 0, done.stdout
