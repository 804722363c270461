"""csrc/math64.cuh compiled for the host: division and square root are correctly
rounded for every result that the single-precision reciprocals may give (one
ulp either way), and exp, sin, cos stay within 0.6 ulp."""
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2408_09662_gb300", "csrc")

HOST = r"""
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <random>
#define CS_MATH_HOST
#define __device__
#define __noinline__ __attribute__((noinline))
#define __forceinline__ inline
typedef uint32_t u32; typedef uint64_t u64;
template <class T, class F> static T as(F f) { T t; memcpy(&t, &f, sizeof t); return t; }
static u32 __umulhi(u32 a, u32 b) { return (u64)a * b >> 32; }
static u32 __funnelshift_l(u32 lo, u32 hi, u32 s) { s &= 31; return s ? hi << s | lo >> (32 - s) : hi; }
static u32 __funnelshift_r(u32 lo, u32 hi, u32 s) { s &= 31; return s ? lo >> s | hi << (32 - s) : lo; }
static int __clz(int x) { return x ? __builtin_clz((u32)x) : 32; }
static int __double2hiint(double d) { return (int)(as<u64>(d) >> 32); }
static int __double2loint(double d) { return (int)as<u64>(d); }
static double __hiloint2double(int h, int l) { return as<double>((u64)(u32)h << 32 | (u32)l); }
static float __uint_as_float(u32 u) { return as<float>(u); }
static u32 __float_as_uint(float f) { return as<u32>(f); }
static float __fmaf_rd(float a, float b, float c) {
  double p = (double)a * b + c; float r = (float)p; return r > p ? nextafterf(r, -INFINITY) : r;
}
static u64 cs_shr64(u64 a, u32 s) { return s > 63 ? 0 : a >> s; }
static u64 cs_shl64(u64 a, u32 s) { return s > 63 ? 0 : a << s; }
static int off;
static float nudge(double v) { float r = (float)v; return off ? nextafterf(r, off > 0 ? 9.f : 0.f) : r; }
static float cs_rcpf(float x) { return nudge(1.0 / x); }
static float cs_rsqrtf(float x) { return nudge(1.0 / sqrt((double)x)); }
#include "math64.cuh"
static std::mt19937_64 g(1);
static double bits(int lo, int hi) {
  u64 m = g(), low = (1ull << g() % 52) - 1;
  if (g() % 4 == 0) m &= ~low; else if (g() % 4 == 0) m |= low;
  return as<double>((g() & 1ull << 63) | (u64)(lo + g() % (hi - lo + 1)) << 52 | (m & 0xfffffffffffffull));
}
template <class F, class R> static double worst(F f, R r, double lo, double hi) {
  double w = 0;
  for (int i = 0; i < 200000; ++i) {
    double x = lo + (hi - lo) * (g() >> 11) * 0x1p-53, y = f(x);
    long double v = r((long double)x); int e; frexpl(v, &e);
    w = fmax(w, (double)fabsl((y - v) / ldexpl(1, e - 53)));
  }
  return w;
}
int main() {
  long bad = 0;
  for (off = -1; off <= 1; ++off)
    for (int i = 0; i < 400000; ++i) {
      double a = bits(1, 2046), b = bits(400, 1600), s = fabs(bits(1, 2046));
      if (i % 8 == 0) a = b * (1 + (int)(g() % 5 - 2) * 0x1p-52);
      if (i % 8 == 1) { s = 1 + g() % 1000 * 0x1p-52; s *= s; }
      bad += as<u64>(cs_div64(a, b)) != as<u64>(a / b);
      bad += as<u64>(cs_sqrt64(s)) != as<u64>(sqrt(s));
    }
  off = 0;
  double w = fmax(worst(cs_exp64, expl, -30, 2), worst(cs_exp64, expl, -708, 708));
  w = fmax(w, fmax(worst(cs_sin64, sinl, -10, 10), worst(cs_cos64, cosl, -10, 10)));
  w = fmax(w, fmax(worst(cs_sin64, sinl, -2e5, 2e5), worst(cs_cos64, cosl, -2e5, 2e5)));
  printf("%ld %.4f\n", bad, w);
}
"""


def test_host_build_of_the_fp64_functions(tmp_path):
    if os.uname().machine != "x86_64":
        pytest.skip("the extended-precision reference functions are the x87 ones")
    src = tmp_path / "host.cpp"
    src.write_text(HOST)
    exe = str(tmp_path / "host")
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-w", "-I", CSRC, "-o", exe, str(src)], check=True)
    bad, worst = subprocess.run([exe], check=True, capture_output=True, text=True).stdout.split()
    assert int(bad) == 0
    assert float(worst) <= 0.6


# the forms with several results or a divisor used again, against the plain ones
FORMS = r"""
int main() {
  long bad = 0;
  const double edge[] = {0.0, -0.0, INFINITY, -INFINITY, NAN, 5e-324, -5e-324, 0x1p-1022, 0x1.fffffffffffffp-1023, 0x1p-510,
                         0x1p-509, 0x1.fffffffffffffp-510, 0x1.fffffffffffffp+512, 0x1p+513, 0x1.fffffffffffffp+1023, 1.0,
                         -3.0, 0x1.fffffffffffffp+0, 0x1.0000000000001p+0};
  auto same = [](double a, double b) { return as<u64>(a) == as<u64>(b) || (std::isnan(a) && std::isnan(b)); };
  auto divide = [&](double a, double c, double b) {
    const u64 r = cs_recip64(b);
    double p, q;
    cs_divr64x2(a, c, b, r, p, q);
    bad += !same(cs_divr64(a, b, r), a / b) + !same(p, a / b) + !same(q, c / b);
    u64 u = as<u64>(b) & 0xfffffffffffffull;       // the reciprocal of a constant, as the generator gives it
    u = u ? (u64)(((unsigned __int128)1 << 116) / (u | 1ull << 52)) : ~0ull;
    bad += !same(cs_divr64(a, b, u), a / b);
  };
  for (off = -1; off <= 1; ++off) {
    for (double a : edge)
      for (double c : edge)
        for (double b : edge) divide(a, c, b);
    for (int i = 0; i < 300000; ++i) {
      double a = bits(1, 2046), c = bits(500, 1500), b = bits(400, 1600);
      if (i % 4 == 0) a = b * (1 + (int)(g() % 5 - 2) * 0x1p-52);
      if (i % 4 == 1) c = b * (double)(g() % (1 << 20));
      divide(a, c, b);
    }
  }
  off = 0;
  auto trig = [&](double x) {
    double s, c;
    cs_sincos64(x, s, c);
    bad += !same(s, cs_sin64(x)) + !same(c, cs_cos64(x));
  };
  for (double x : edge) trig(x);
  for (double x : {0x1p-27, 0x1p+18, 0.5}) for (double y : {x, nextafter(x, 0.0), nextafter(x, 1e9)}) { trig(y); trig(-y); }
  for (int i = 0; i < 400000; ++i) trig(bits(980, 1042));
  for (int k = 1; k < 160000; ++k) {               // next to multiples of pi/2
    const double x = (double)(k * 1.57079632679489661923132169163975144L);
    trig(x); trig(-x); trig(nextafter(x, 0.0)); trig(nextafter(x, 1e9));
  }
  printf("%ld\n", bad);
}
"""


def test_forms_with_several_results_equal_the_plain_ones(tmp_path):
    if os.uname().machine != "x86_64":
        pytest.skip("the extended-precision reference functions are the x87 ones")
    (tmp_path / "host.cpp").write_text(HOST[:HOST.index("int main()")] + FORMS)
    exe = str(tmp_path / "host")
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-w", "-I", CSRC, "-o", exe, str(tmp_path / "host.cpp")],
                   check=True)
    assert int(subprocess.run([exe], check=True, capture_output=True, text=True).stdout) == 0
