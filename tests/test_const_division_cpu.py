"""FP32 division by a constant as the generated kernels do it, compiled for the
host: the bits of x / c."""
import re
import subprocess

import pytest

from paper_2408_09662_gb300 import tracer as T
from paper_2408_09662_gb300.api import Function

CONSTANTS = [k / 1000 for k in range(1, 1000) if k not in (125, 250, 500)] + [
    3.0, 5.0, 6.0, 7.0, 10.0, 12.0, 24.0, 49.0, 1.0000001, 1.9999999, 8388609.0, 16777215.0, 16777214.0, 1.1 * 2.0 ** -20]

HOST = r"""
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <random>
typedef uint32_t u32;
template <class T, class F> static T as(F f) { T t; memcpy(&t, &f, sizeof t); return t; }
#define __device__
#define __forceinline__ inline
static float __fmul_rn(float a, float b) { return a * b; }
static float __int_as_float(int i) { return as<float>(i); }
static u32 __float_as_uint(float f) { return as<u32>(f); }
static float __uint_as_float(u32 u) { return as<float>(u); }
FUNCTIONS
static const struct { float c; float (*divide)(float); } cs[] = { TABLE };
static std::mt19937_64 g(1);
int main() {
  for (auto& k : cs) {
    long bad = 0;
    float at = 0;
    auto check = [&](float x) {
      const float y = k.divide(x), w = x / k.c;
      if (as<u32>(y) != as<u32>(w) && !(std::isnan(y) && std::isnan(w))) { ++bad; at = x; }
    };
    ARGUMENTS
    if (bad) printf("c = %.9g: %ld, one at x = %.9g\n", k.c, bad, at);
  }
}
"""

EVERY_EXPONENT = "for (int i = 0; i < 20000; ++i) { float x = as<float>((u32)g()); if (KEEP) check(x); }"
# |x| up to the largest finite value, around the least whose quotient overflows
OVERFLOW = ("for (int i = -40; i <= 40; ++i) { const float x = (float)((double)k.c * 0x1p128);"
            "  const u32 b = std::isfinite(x) ? as<u32>(x) : 0x7f7fffe0u; check(as<float>(b + i)); check(-as<float>(b + i)); }"
            "for (u32 i = 0; i < 64; ++i) { check(as<float>(0x7f800000u - i)); check(as<float>(0xff800000u - i)); }"
            "check(0.0f); check(-0.0f); check(NAN);")


def differences(tmp_path, arguments):
    (x,) = T.Graph().symbols(1)
    ir = T.Function([("x", [x])], [("y", [x / c for c in CONSTANTS])]).to_ir()
    src = Function(ir, dtype="f32", cache_dir=None).source()
    functions = re.findall(r"static __device__ __forceinline__ float cs_divc2?_f\(.*?\n}\n", src, flags=re.S)
    calls = re.findall(r" (cs_divc2?_f)\(v\d+, (\S+), (.*)\);", src)
    assert len(calls) == len(CONSTANTS) and len({c[0] for c in calls}) == 2
    text = HOST.replace("FUNCTIONS", "".join(functions)).replace("ARGUMENTS", arguments)
    text = text.replace("TABLE", ", ".join(
        f"{{{c}, [](float x) {{ return {f}(x, {c}, {rest}); }}}}" for f, c, rest in calls))
    (tmp_path / "host.cpp").write_text(text)
    exe = str(tmp_path / "host")
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-w", "-o", exe, str(tmp_path / "host.cpp")], check=True)
    return subprocess.run([exe], check=True, capture_output=True, text=True).stdout


def test_normal_quotients_and_overflow(tmp_path):
    arguments = OVERFLOW + EVERY_EXPONENT.replace("KEEP", "std::fabs((double)x / k.c) >= 0x1p-126")
    assert differences(tmp_path, arguments) == ""


# x whose quotients are subnormal: every exponent, and next to halves of the grid
SUBNORMAL = ("for (int i = 0; i < 4000; ++i) { const double h = ((double)(g() % (1u << (1 + g() % 23))) + 0.5) * 0x1p-149;"
             "  const float x = (float)(h * k.c); check(x); check(-std::nextafterf(x, 1)); check(std::nextafterf(x, -1)); }"
             "for (int i = 0; i < 4000; ++i) check(as<float>((u32)(g() % as<u32>(std::fmax(k.c, 0x1p-20f) * 0x1p-125f))));"
             "for (u32 i = 0; i < 3000; ++i) check(as<float>(i));")


def test_subnormal_quotients(tmp_path):
    assert differences(tmp_path, SUBNORMAL + EVERY_EXPONENT.replace("KEEP", "true")) == ""


@pytest.mark.parametrize("ways", [0, 2])
@pytest.mark.parametrize("dtype,least,most", [("f64", -1022, 1022), ("f32", -126, 126)])
def test_division_by_a_power_of_two_is_a_multiply(dtype, least, most, ways):
    """Where the reciprocal is a normal number: exact, and free to join an add."""
    (x,) = T.Graph().symbols(1)
    k = [2.0, -0.25, 2.0 ** least, 2.0 ** most]
    src = Function(T.Function([("x", [x])], [("y", [x / c for c in k])]).to_ir(), dtype=dtype, ways=ways, cache_dir=None).source()
    suffix = "f" if dtype == "f32" else ""
    for r in ("0x1p-1", "-0x1p+2", f"0x1p{-least:+d}", f"0x1p{-most:+d}"):
        assert re.search(r"(mul_rn\(v\w+, | \* )" + re.escape(f"({r}{suffix})"), src), r
    assert not re.search(r"= v\w+ / |cs_div\w*\(v", src)
    beyond = Function(T.Function([("x", [x])], [("y", [x / 2.0 ** (least - 1)])]).to_ir(), dtype=dtype, ways=ways, cache_dir=None)
    assert not re.search(r"(mul_rn\(v\w+, | \* )\(0x", beyond.source())
