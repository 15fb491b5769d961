"""Host check of csrc/roots.cuh: the reciprocal square root after one Newton step, and the
square root formed from a reciprocal, for every estimate within the bound that they are
given (2 ulp in FP32, the hardware's; 1 ulp for the reciprocal of the root).

Bounds, in units u of half an ulp at the larger mantissas (2^-24, 2^-53 relative): the step
rounds x y (u / 2 in the result) and the result itself (half an ulp), and leaves 1.5 e^2 of
an estimate's error e <= 4 u: 1 ulp + 1e-5.  The root's step leaves e^2 / 2 + e d of the
product's error e <= 3 u and the reciprocal's d <= 2 u: half an ulp + 1e-6 in FP32, and the
2^-10 ulp that a long double resolves in FP64."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1903_10134_gb300", "csrc")

PROGRAM = r"""
#include "roots.cuh"
#include <cstdio>
#include <random>
using namespace mdpd;

template <typename T> static T moved(T y, int ulps)
{
    for (; ulps > 0; --ulps) y = std::nextafter(y, (T)INFINITY);
    for (; ulps < 0; ++ulps) y = std::nextafter(y, (T)0);
    return y;
}
template <typename T> static double ulps(T got, long double want)
{
    const T w = (T)want;
    const long double ulp = (long double)std::nextafter(w, (T)INFINITY) - (long double)w;
    return (double)(std::fabs((long double)got - want) / ulp);
}

int main()
{
    std::mt19937_64 rng(7);
    std::uniform_real_distribution<double> expo(std::log(1e-30), std::log(1e3)), unit(0.0, 1.0);
    double step = 0, root = 0, root64 = 0;
    for (int i = 0; i < 400000; ++i) {
        const double q = i % 2 ? std::exp(expo(rng)) : unit(rng) + 1e-12;
        const float x = (float)q;
        const long double r = std::sqrt((long double)x);
        for (int k = -2; k <= 2; ++k)
            step = std::fmax(step, ulps(inv_sqrt_step(x, moved((float)(1 / r), k)), 1 / r));
        for (int k = -1; k <= 1; ++k)
            root = std::fmax(root, ulps(sqrt_from(x, moved((float)(1 / r), k)), r));
        const long double r64 = std::sqrt((long double)q);
        for (int k = -1; k <= 1; ++k)
            root64 = std::fmax(root64, ulps(sqrt_from(q, moved((double)(1 / r64), k)), r64));
    }
    std::printf("%.9g %.9g %.9g\n", step, root, root64);
    return 0;
}
"""


@pytest.mark.skipif(shutil.which("g++") is None, reason="no host compiler")
def test_roots_within_their_bounds(tmp_path):
    src, exe = tmp_path / "roots.cpp", tmp_path / "roots"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-x", "c++", "-I", CSRC, str(src),
                    "-o", str(exe), "-lm"], check=True)
    step, root, root64 = map(float, subprocess.run([str(exe)], check=True, capture_output=True,
                                                   text=True).stdout.split())
    assert step <= 1.0 + 1e-5
    assert root <= 0.5 + 1e-6
    assert root64 <= 0.5 + 2.0 ** -10
