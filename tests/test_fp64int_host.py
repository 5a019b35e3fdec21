"""csrc/fp64int.cuh against the language's own conversions and comparisons, with
the header compiled for the host and the five bit casts it uses written out:
ties, subnormals, both ends of FP32's range, infinities and random bit patterns.
Equality is exact (NaN: NaN)."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

STUB = r"""
#pragma once
#include <stdint.h>
#include <string.h>
#define __device__
#define __forceinline__ inline
template <class A, class B> inline A bits_of(B b) { A a; memcpy(&a, &b, sizeof a); return a; }
inline long long __double_as_longlong(double x) { return bits_of<long long>(x); }
inline int __double2hiint(double x) { return (int)(bits_of<uint64_t>(x) >> 32); }
inline int __double2loint(double x) { return (int)bits_of<uint64_t>(x); }
inline double __hiloint2double(int h, int l) { return bits_of<double>((uint64_t)(uint32_t)h << 32 | (uint32_t)l); }
inline uint32_t __float_as_uint(float f) { return bits_of<uint32_t>(f); }
inline float __uint_as_float(uint32_t u) { return bits_of<float>(u); }
"""

MAIN = r"""
#include <math.h>
#include <stdio.h>
#include <vector>
#include "fp64int.cuh"
using namespace ifci;
static long long bad = 0;
static void narrow(double x) {
    const float a = d2f(x), b = (float)x;
    if (isnan(b) ? !isnan(a) : __float_as_uint(a) != __float_as_uint(b)) { if (bad++ < 5) printf("d2f %a: %a, %a\n", x, a, b); }
}
static void widen(uint32_t u) {
    const float f = __uint_as_float(u);
    const double a = f2d(f), b = (double)f;
    if (isnan(b) ? !isnan(a) : dbits(a) != dbits(b)) { if (bad++ < 5) printf("f2d %a: %a, %a\n", f, a, b); }
}
int main() {
    uint64_t s = 88172645463325252ull;
    auto rnd = [&]() { s ^= s << 13; s ^= s >> 7; s ^= s << 17; return s; };
    for (int e = 0; e < 2048; e++) {
        // mantissas at, just below and just above a tie of the 29 bits that go, even and odd above it
        for (uint64_t keep : {0ull, 1ull, 0x3FFFFFull, 0x7FFFFEull, 0x7FFFFFull})
            for (long long low : {0ll, 1ll, 0x0FFFFFFFll, 0x10000000ll, 0x10000001ll, 0x1FFFFFFFll})
                for (uint64_t sign : {0ull, 1ull})
                    narrow(bits_of<double>(sign << 63 | (uint64_t)e << 52 | keep << 29 | (uint64_t)low));
        for (int k = 0; k < 500; k++) narrow(bits_of<double>((rnd() & ~(0x7FFull << 52)) | (uint64_t)e << 52));
    }
    for (uint32_t e = 0; e < 256; e++)
        for (int k = 0; k < 2000; k++) {
            const uint32_t m = k == 0 ? 0 : k == 1 ? 1 : k == 2 ? 0x7FFFFF : (uint32_t)rnd() & 0x7FFFFF;
            widen(e << 23 | m);
            widen(0x80000000u | e << 23 | m);
        }
    std::vector<double> v = {0.0, 5e-324, 2.2250738585072014e-308, 1.0, 1.0000000000000002, 1.7976931348623157e308, INFINITY};
    for (int k = 0; k < 300; k++) { const double x = bits_of<double>(rnd()); if (!isnan(x)) v.push_back(fabs(x)); }
    for (size_t i = 0, n = v.size(); i < n; i++) v.push_back(-v[i]);
    for (double x : v) {
        if (bits_of<double>(dmag(x)) != fabs(x) || dbits(dflip(x, 0x80000000u)) != dbits(-x) || dbits(dflip(x, 0u)) != dbits(x)) bad++;
        for (double y : v)
            if (x != y && (dkey(x) < dkey(y)) != (x < y)) { if (bad++ < 5) printf("dkey %a %a\n", x, y); }
    }
    if (!(dkey(-0.0) < dkey(0.0))) bad++;
    printf("%lld wrong\n", bad);
    return bad != 0;
}
"""


def test_integer_forms_give_the_same_results(tmp_path):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no host compiler")
    (tmp_path / "cuda_runtime.h").write_text(STUB)
    (tmp_path / "main.cpp").write_text(MAIN)
    exe = str(tmp_path / "check")
    subprocess.run([cxx, "-std=c++17", "-O1", "-I", str(tmp_path), "-I",
                    os.path.join(ROOT, "paper_2307_10675_gb300", "csrc"), str(tmp_path / "main.cpp"), "-o", exe],
                   check=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
