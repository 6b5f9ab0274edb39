"""The integer conversions of csrc/dd.cuh give the bits of the plain casts.

f32_of(v) = (float)v and dd_split(v) = dd(v), over random doubles of every
exponent, both signs, the neighbours of FP32 rounding ties and of powers of
two, subnormals, zeros, infinities and NaN. The header is compiled unchanged
by the host C++ compiler, with a stub for the CUDA qualifiers.
"""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1601_05970_gb300", "csrc")

STUB = """#pragma once
#define __device__
#define __host__
#define __forceinline__ inline
#define __align__(n) alignas(n)
"""

HARNESS = r"""
#include <cstdio>
#include <cstdint>
#include <cstring>
#include <random>
#include "dd.cuh"
using namespace fftg;

static double make(uint64_t u) { double v; std::memcpy(&v, &u, 8); return v; }
static uint32_t b32(float f) { uint32_t u; std::memcpy(&u, &f, 4); return u; }
static long bad = 0, seen = 0;

static void one(uint64_t u) {
    const double v = make(u);
    const float a = f32_of(v), b = (float)v;
    const dd s = dd_split(v), t(v);
    const bool nan = v != v;
    ++seen;
    bool ok = nan ? a != a : b32(a) == b32(b);
    // lo of an infinity is NaN either way
    ok = ok && (nan ? s.hi != s.hi : b32(s.hi) == b32(t.hi));
    ok = ok && ((t.lo != t.lo) ? s.lo != s.lo : b32(s.lo) == b32(t.lo));
    if (!ok && ++bad < 20) std::printf("%016llx\n", (unsigned long long)u);
}

int main() {
    std::mt19937_64 g(7);
    for (uint64_t e = 0; e < 2048; ++e)
        for (int sgn = 0; sgn < 2; ++sgn) {
            const uint64_t top = (uint64_t)sgn << 63 | e << 52;
            for (int k = 0; k < 200; ++k) {
                const uint64_t m = g() >> 12;
                one(top | m);
                // about a tie of the FP32 rounding, even and odd last bits
                const uint64_t tie = (m & ~0x1fffffffull) | 0x10000000ull;
                one(top | tie);
                one(top | (tie - 1));
                one(top | (tie + 1));
                one(top | (m & ~0x1fffffffull));
                one(top | (m >> (k % 52)));
            }
            one(top);
            one(top | 1);
            one(top | 0xfffffffffffffull);
            one(top | 0xfffffe0000000ull);
            one(top | 0xffffff0000000ull);
        }
    std::printf("%ld values, %ld differ\n", seen, bad);
    return bad != 0;
}
"""


def test_conversions_give_the_bits_of_the_casts(tmp_path):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no host compiler")
    (tmp_path / "cuda_runtime.h").write_text(STUB)
    (tmp_path / "t.cpp").write_text(HARNESS)
    exe = str(tmp_path / "t")
    subprocess.run([cxx, "-std=c++17", "-O2", "-ffp-contract=off", "-I" + str(tmp_path), "-I" + CSRC,
                    str(tmp_path / "t.cpp"), "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
