"""Compiles a device header of csrc/ that needs nothing but bit-cast and rounding
intrinsics (written here in C++) with a test program, and runs it."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2404_08849_gb300", "csrc")
SHIM = r"""
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <limits>
#include <random>
#define __device__
#define __forceinline__ inline
static uint64_t bits(double x) { uint64_t u; memcpy(&u, &x, 8); return u; }
static uint32_t bits(float x) { uint32_t u; memcpy(&u, &x, 4); return u; }
static double real(uint64_t u) { double x; memcpy(&x, &u, 8); return x; }
static float real32(uint32_t u) { float x; memcpy(&x, &u, 4); return x; }
static int __double2hiint(double x) { return (int)(bits(x) >> 32); }
static int __double2loint(double x) { return (int)bits(x); }
static double __hiloint2double(int h, int l) { return real(((uint64_t)(uint32_t)h << 32) | (uint32_t)l); }
static long long __double_as_longlong(double x) { return (long long)bits(x); }
static double __longlong_as_double(long long x) { return real((uint64_t)x); }
static float __fsub_rn(float a, float b) { return a - b; }
static float __fadd_rn(float a, float b) { return a + b; }
// the same number, or both NaN
static bool same(double a, double b) { return bits(a) == bits(b) || (std::isnan(a) && std::isnan(b)); }
static bool same(float a, float b) { return bits(a) == bits(b) || (std::isnan(a) && std::isnan(b)); }
"""
# what forms.cuh takes from common.cuh, as plain operations
PLAIN = """
static double f2d(float f) { return (double)f; }
static double sub_near(double a, double b) { return a - b; }
// any reciprocal within one ulp
static float rcp_approx(float x) {
    static uint32_t n = 0;
    const float y = 1 / x;
    if (!std::isfinite(x) || x == 0) return y;
    n = n * 1664525u + 1013904223u;
    const float z = n >> 30 == 0 ? std::nextafter(y, -INFINITY) : n >> 30 == 1 ? std::nextafter(y, INFINITY) : y;
    return std::fabs((double)z - 1.0 / x) <= std::fabs((double)std::nextafter(y, 2 * y) - y) ? z : y;
}
"""


def run(tmp_path, header, main, shim=""):
    """Numbers that `main` prints, as floats."""
    if shutil.which("g++") is None:
        pytest.skip("g++ not found")
    src = tmp_path / "test.cpp"
    src.write_text(SHIM + shim + '#include "%s"\nusing namespace grist;\n' % os.path.join(CSRC, header) + main)
    exe = tmp_path / "test"
    subprocess.run(["g++", "-std=c++17", "-O2", "-ffp-contract=off", "-o", str(exe), str(src)], check=True)
    return [float(x) for x in subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split()]
