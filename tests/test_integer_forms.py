"""The integer forms of FP64 operations (csrc/common.cuh: sub_near, MulF32)
against the operations themselves, bit for bit, on the host: the functions'
source compiled with the few device intrinsics they use written in C++."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SHIM = r"""
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <random>
using std::min;
#define __device__
#define __forceinline__ inline
static uint64_t bits(double x) { uint64_t u; memcpy(&u, &x, 8); return u; }
static double real(uint64_t u) { double x; memcpy(&x, &u, 8); return x; }
static int __double2hiint(double x) { return (int)(bits(x) >> 32); }
static int __double2loint(double x) { return (int)bits(x); }
static double __hiloint2double(int h, int l) { return real(((uint64_t)(uint32_t)h << 32) | (uint32_t)l); }
static int __clzll(long long x) { return x ? __builtin_clzll(x) : 64; }
static uint32_t __float_as_uint(float f) { uint32_t u; memcpy(&u, &f, 4); return u; }
static uint32_t __funnelshift_l(uint32_t lo, uint32_t hi, uint32_t s) { return s ? (hi << s) | (lo >> (32 - s)) : hi; }
"""
MAIN = r"""
int main() {
    std::mt19937_64 r(7);
    long bad = 0, taken = 0;
    const long n = 3000000;
    for (long i = 0; i < n; i++) {          // a - b: equal, close, one binade apart, any, subnormal
        uint64_t u = r(), v;
        switch (i % 7) {
            case 0: v = u + (int64_t)(r() % 1000) - 500; break;
            case 1: v = u + (int64_t)(r() % (1ull << 53)) - (1ll << 52); break;
            case 2: v = r(); break;
            case 3: v = (u & 0xfff0000000000000ull) | (r() & 0xfffffffffffffull); break;
            case 4: v = ((u + ((r() % 5 - 2) << 52))) ^ (r() & 0xfffffffffffffull); break;
            case 5: v = u; break;
            default:
                u = (u & 0x800fffffffffffffull) | ((r() % 4) << 52);
                v = (u & 0x8000000000000000ull) | (r() & 0x003fffffffffffffull);
        }
        const double a = real(u), b = real(v), x = sub_near(a, b), y = a - b;
        if (!(std::isnan(x) && std::isnan(y)) && bits(x) != bits(y)) bad++;
    }
    for (long i = 0; i < n; i++) {          // w * u: any, physical sizes, ties, zeros
        uint64_t wb = r();
        uint32_t ub = (uint32_t)r();
        if (i % 4 == 1) {
            wb = (wb & 0x800fffffffffffffull) | ((1023ull - 60 + r() % 120) << 52);
            ub = (ub & 0x807fffffu) | ((100 + r() % 60) << 23);
        }
        if (i % 4 == 2) {
            wb = (wb & (~0ull << (r() % 50)) & 0x800fffffffffffffull) | (1023ull << 52);
            ub &= ~0u << (r() % 23);
        }
        if (i % 97 == 0) ub &= 0x80000000u;
        const int e = (int)((wb >> 52) & 0x7ff);
        if (e == 0 || e == 2047) continue;
        float u;
        memcpy(&u, &ub, 4);
        const MulF32 m(real(wb));
        bool ok = true;
        const double x = m.times(u, ok);
        if (!ok) continue;
        taken++;
        if (bits(x) != bits(real(wb) * (double)u)) bad++;
    }
    printf("%ld %ld\n", bad, taken);
    return 0;
}
"""


def test_same_bits_as_the_fp64_operations(tmp_path):
    if shutil.which("g++") is None:
        pytest.skip("g++ not found")
    src = open(os.path.join(ROOT, "paper_2404_08849_gb300", "csrc", "common.cuh")).read()
    sub = src[src.index("__device__ __forceinline__ double sub_near"):]
    sub = sub[:sub.index("\n}\n") + 3]
    mul = src[src.index("struct MulF32 {"):]
    mul = mul[:mul.index("\n};\n") + 4]
    c = tmp_path / "forms.cpp"
    c.write_text(SHIM + sub + mul + MAIN)
    exe = tmp_path / "forms"
    subprocess.run(["g++", "-O2", "-ffp-contract=off", "-o", str(exe), str(c)], check=True)
    bad, taken = (int(x) for x in subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split())
    assert bad == 0
    assert taken > 2000000
