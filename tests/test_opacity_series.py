"""The opacity correction's series against 64-bit arithmetic, on the host: the
functions that the march kernels call, compiled for the CPU, over ratios from a
thousandth to two and opacities up to the cut, and the general formula above it,
for ratios above two, and for opacities of 0 and 1."""
import subprocess

from paper_2501_01628_gb300 import build

HARNESS = r'''
#include <algorithm>
#include <cmath>
#include <cstdio>
#include "vr_device.cuh"
using namespace vr;
int main()
{
    double worst = 0.0, general = 0.0;
    int bad = 0;
    for (int i = 1; i <= 2000; ++i) {
        const float ratio = i / 1000.0f;
        if (ratio == 1.0f) continue;
        const OpacityStep o = opacity_step(ratio, 0.18f);
        if (!(o.cut >= 0.18f && o.cut <= 0.25f)) ++bad;
        for (float most : {0.251f, 1.0f, INFINITY, NAN})
            if (opacity_step(ratio, most).cut != -1.0f) ++bad;
        for (int j = -2000; j <= 2000; ++j) {
            const float a = o.cut * (j / 2000.0f);
            const double want = -std::expm1(static_cast<double>(ratio) * std::log1p(-static_cast<double>(a)));
            const float got = dev::corrected_opacity<kOpacitySeries>(a, o), was = -expm1f(ratio * log1pf(-a));
            if (j == 0) {
                if (got != 0.0f || std::signbit(got)) ++bad;
                continue;
            }
            worst = std::max(worst, std::fabs(got - want) / std::fabs(want));
            general = std::max(general, std::fabs(was - want) / std::fabs(want));
        }
        for (float a : {0.3f, 0.5f, 0.99f, 1.0f})
            if (dev::corrected_opacity<kOpacitySeries>(a, o) != -expm1f(ratio * log1pf(-a))) ++bad;
    }
    for (float ratio : {2.001f, 4.0f, 37.0f, 1e6f}) {
        const OpacityStep o = opacity_step(ratio, 0.1f);
        for (float a : {0.0f, 1e-6f, 0.1f, 0.25f, 1.0f})
            if (dev::corrected_opacity<kOpacitySeries>(a, o) != -expm1f(ratio * log1pf(-a))) ++bad;
    }
    const double u = 1.0 / 16777216.0;
    std::printf("%.3f %.3f %d\n", worst / u, general / u, bad);
}
'''


def test_series_against_64_bits(tmp_path):
    src = tmp_path / "opacity.cu"
    src.write_text(HARNESS)
    exe = tmp_path / "opacity"
    subprocess.run([build.nvcc(), *build.ARCH, "-O2", "-std=c++17",
                    "-I", build.CSRC, "-o", str(exe), str(src)], check=True, timeout=600)
    worst, general, bad = subprocess.run([str(exe)], check=True, capture_output=True, text=True,
                                         timeout=120).stdout.split()
    print(worst, general)
    assert int(bad) == 0
    # in units of 2^-24: the last sum's rounding, that of ratio * a (at most 8/7 of
    # the result), the terms left out (1/8), and the roundings of a^2, of the inner
    # sum and of its coefficients, weighted by |a^2 s| <= 1/7 of the result
    assert float(worst) <= 2.7
