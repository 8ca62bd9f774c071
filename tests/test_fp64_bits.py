"""The FP64 comparisons that csrc/device_common.cuh makes on the bits of a
double, compiled for the host: they decide as the comparisons do, for zeros of
both signs, the ends of every range, infinities and NaN, and their integer
arithmetic is defined for all of them (the build traps on signed overflow)."""
import os
import subprocess

from paper_2507_03366_gb300 import build

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SOURCE = r"""
#include <cuda_runtime.h>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <limits>
using std::fma; using std::fmax; using std::isfinite; using std::sqrt;
static inline float __fmul_rn(float a, float b) { return a * b; }
static inline double __dadd_rn(double a, double b) { return a + b; }
static inline float __fdividef(float a, float b) { return a / b; }
static inline long long __double_as_longlong(double x) { long long r; std::memcpy(&r, &x, 8); return r; }
static inline int __double2hiint(double x) { return (int)(__double_as_longlong(x) >> 32); }
template <class T> static inline T __ldcg(const T* p) { return *p; }
#include "device_common.cuh"

static bool same(double a, double b) { return std::memcmp(&a, &b, 8) == 0; }

int main() {
    typedef std::numeric_limits<double> L;
    const double m[] = {0.0, L::denorm_min(), 3e-310, L::min(), 1e-17, 0.5, std::nextafter(1.0, 0.0), 1.0,
                        std::nextafter(1.0, 2.0), 3.0, 1e300, L::max(), L::infinity(), L::quiet_NaN(),
                        L::signaling_NaN()};
    int bad = 0;
    for (double a : m)
        for (int s = 0; s < 2; ++s) {
            volatile double v = s ? -a : a;
            const double x = v;
            bad += eulbfs::positive(x) != (x > 0.0);
            bad += eulbfs::negative(x) != (x < 0.0);
            bad += eulbfs::is_finite(x) != (bool)isfinite(x);
            const double c = x < 0.0 ? 0.0 : (x > 1.0 ? 1.0 : x), g = eulbfs::clamp01(x);
            bad += std::isnan(c) ? !std::isnan(g) : !same(g, c);
        }
    std::printf("%d\n", bad);
    return 0;
}
"""


def test_bit_comparisons_decide_as_the_comparisons(tmp_path):
    src, exe = tmp_path / "bits.cpp", tmp_path / "bits"
    src.write_text(SOURCE)
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(build.nvcc()))), "include")
    subprocess.run(["g++", "-std=c++17", "-O1", "-fsanitize=signed-integer-overflow",
                    "-fsanitize-undefined-trap-on-error", "-I", cuda, "-I", os.path.join(ROOT, "include"), "-I",
                    os.path.join(ROOT, "paper_2507_03366_gb300", "csrc"), str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0 and r.stdout.split() == ["0"]
