"""The formation's double-float sigmoid (csrc/sigmoid.cuh) compiled for the host,
every operation with its single rounding, against long double: the relative
error of the pair from the threshold up, and opacities and App. C.1 positions
equal to size * sigmoid rounded once over the whole range, sizes that no float
holds among them. (The formula (tanh x + 1) / 2, which FP64 loses digits in for
negative x, is no reference below x = -4.)"""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2403_08551_gb300", "csrc")

MAIN = """
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <random>
#define __device__
#define __forceinline__ inline
struct float2 { float x, y; };
static float __fmul_rn(float a, float b) { return a * b; }
static float __fadd_rn(float a, float b) { return a + b; }
static float __fsub_rn(float a, float b) { return a - b; }
static float __fmaf_rn(float a, float b, float c) { return std::fma(a, b, c); }
static float __frcp_rn(float a) { return 1.0f / a; }
static double __dmul_rn(double a, double b) { return a * b; }
static int __float2int_rn(float a) { return (int)std::nearbyint(a); }
static float __int2float_rz(int a) { float f = (float)a; return (double)f > (double)a ? std::nextafter(f, 0.0f) : f; }
static float __int_as_float(int a) { float f; std::memcpy(&f, &a, 4); return f; }
using std::fabs; using std::fmin; using std::rint;
#include "sigmoid.cuh"
using namespace gi;
static long double ref(long double t) {
    const long double e = std::exp(-std::fabs(t));
    return (t < 0 ? e : 1.0L) / (1.0L + e);
}
int main() {
    std::mt19937_64 g(3);
    auto uni = [&](float lo, float hi) { return std::uniform_real_distribution<float>(lo, hi)(g); };
    long double worst = 0;
    const float ends[] = {kSigmoidMin, -16.f, -8.f, -4.f, 0.f, 4.f, 16.f, 60.f};
    for (int r = 0; r < 7; ++r)
        for (int i = 0; i < 400000; ++i) {
            const float t = uni(ends[r], ends[r + 1]);
            float hi, lo;
            sigmoid_dd(t, hi, lo);
            worst = std::fmax(worst, std::fabs(((long double)hi + lo) / ref(t) - 1.0L));
        }
    if (worst > std::ldexp(1.0L, -42) * 0.8123L) std::printf("error 2^%.2f\\n", (double)std::log2(worst));  // 2^-42.3
    long bad = 0;
    for (float hi : {4.f, 30.f, 110.f})
        for (int i = 0; i < 300000; ++i) {
            const float t = uni(-hi, hi);
            bad += opacity_of(t) != (float)ref(t);
        }
    if (bad) std::printf("%ld opacities\\n", bad);
    for (int size : {1, 517, 2040, 65535, 16777217, 2147483585, 2147483647}) {
        bad = 0;
        for (float hi : {1.f, 4.f, 12.f, 45.f})
            for (int i = 0; i < 100000; ++i) {
                const float x = uni(-hi, hi);
                bad += raw_position(x, size) != (float)((long double)size * ref(2.0L * x));
            }
        if (bad) std::printf("size %d: %ld positions\\n", size, bad);
    }
    const float inf = INFINITY;
    if (raw_position(inf, 517) != 517.f || raw_position(-inf, 517) != 0.f || raw_position(NAN, 517) == raw_position(NAN, 517) ||
        opacity_of(inf) != 1.f || opacity_of(-inf) != 0.f || opacity_of(-0.f) != 0.5f)
        std::puts("limits");
    return 0;
}
"""


@pytest.mark.skipif(shutil.which("g++") is None, reason="no g++")
def test_error_and_rounding(tmp_path):
    (tmp_path / "main.cpp").write_text(MAIN)
    exe = tmp_path / "main"
    subprocess.run(["g++", "-std=c++17", "-O1", "-ffp-contract=off",
                    "-fsanitize=float-cast-overflow,signed-integer-overflow", "-fsanitize-undefined-trap-on-error",
                    "-x", "c++", "-I", CSRC, str(tmp_path / "main.cpp"),
                    "-o", str(exe)], check=True)
    assert subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout == ""
