"""Integer sums of spread forces (spread_sum.h), compiled with g++: the forces
of a sphere's markers, spread with the 4-point kernel, summed per cell in
integers, in FP32 and in FP64. Whatever the components' sizes against each
other, the integer sums are no further from FP64 than FP32 ones, and none
leaves 31 bits."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1906_05448_gb300", "csrc")

HARNESS = r"""
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <random>
#include <vector>
#include "spread_sum.h"
static double peskin(double r) {
    const double a = std::fabs(r);
    if (a <= 1) return (3 - 2 * a + std::sqrt(1 + 4 * a - 4 * a * a)) / 8;
    if (a <= 2) return (5 - 2 * a - std::sqrt(-7 + 12 * a - 4 * a * a)) / 8;
    return 0;
}
int main(int argc, char **argv) {
    const double RL = atof(argv[1]), ratio = atof(argv[2]);
    std::mt19937 rng(atoi(argv[3]));
    std::uniform_real_distribution<double> uni(0, 1);
    std::normal_distribution<double> nor;
    const double pi = 3.14159265358979323846, ga = pi * (3 - std::sqrt(5.0));
    const int n = (int)std::floor(pi / 3 * (12 * RL * RL + 1) + 0.5), W = 2 * (int)std::ceil(RL) + 6;
    const double c[3] = {uni(rng) + W / 2 - 1, uni(rng) + W / 2 - 1, uni(rng) + W / 2 - 1};
    std::vector<float> F(3 * n);
    for (int l = 0; l < n; l++)
        for (int d = 0; d < 3; d++) F[3 * l + d] = (float)(0.01 * (d ? ratio : 1.0) * nor(rng));
    float s[3];
    for (int d = 0; d < 3; d++) {
        float m = 0;
        for (int l = 0; l < n; l++) m = std::fmax(m, std::fabs(F[3 * l + d]));
        s[d] = lbmgb::spread_scale(m);
    }
    std::vector<double> ex(3 * W * W * W);
    std::vector<float> f32(ex.size());
    std::vector<long long> in(ex.size());
    for (int l = 0; l < n; l++) {
        const double z = 1 - (2.0 * l + 1) / n, r = std::sqrt(1 - z * z);
        const double X[3] = {c[0] + RL * r * std::cos(ga * l), c[1] + RL * r * std::sin(ga * l), c[2] + RL * z};
        float ph[3][4];
        int b[3];
        for (int d = 0; d < 3; d++) {
            b[d] = (int)std::floor(X[d]) - 1;
            for (int o = 0; o < 4; o++) ph[d][o] = (float)peskin(b[d] + o - X[d]);
        }
        for (int k = 0; k < 64; k++) {
            const float w = ph[0][k & 3] * ph[1][(k >> 2) & 3] * ph[2][k >> 4];
            const size_t i = (size_t)(b[0] + (k & 3)) + W * ((b[1] + ((k >> 2) & 3)) + (size_t)W * (b[2] + (k >> 4)));
            for (int d = 0; d < 3; d++) {
                const float t = F[3 * l + d] * w;
                ex[3 * i + d] += (double)F[3 * l + d] * w;
                f32[3 * i + d] += t;
                in[3 * i + d] += lbmgb::spread_term(t, s[d]);
            }
        }
    }
    double e32[3] = {0, 0, 0}, ei[3] = {0, 0, 0};
    for (size_t i = 0; i < ex.size(); i++) {
        const int d = (int)(i % 3);
        if (in[i] > 2147483647LL || in[i] < -2147483647LL) return 1;
        e32[d] += std::pow(f32[i] - ex[i], 2);
        ei[d] += std::pow((lbmgb::spread_few(n) ? f32[i] : lbmgb::spread_value((int)in[i], s[d])) - ex[i], 2);
    }
    for (int d = 0; d < 3; d++) std::printf("%.3e %.3e ", std::sqrt(e32[d]), std::sqrt(ei[d]));
    return 0;
}
"""


@pytest.fixture(scope="module")
def exe(tmp_path_factory):
    if shutil.which("g++") is None:
        pytest.skip("no g++")
    d = tmp_path_factory.mktemp("spread")
    (d / "h.cpp").write_text(HARNESS)
    subprocess.run(["g++", "-O1", "-ffp-contract=off", "-std=c++17", "-I", CSRC, str(d / "h.cpp"), "-o", str(d / "h")],
                   check=True)
    return str(d / "h")


@pytest.mark.parametrize("ratio", [1.0, 1e-2, 1e-5])
@pytest.mark.parametrize("RL", [0.1, 0.6, 1.1, 2.3, 3.6, 6.3])
def test_integer_sums_are_no_worse_than_fp32(exe, RL, ratio):
    total = [0.0] * 6
    for seed in range(6):
        r = subprocess.run([exe, str(RL), str(ratio), str(seed)], capture_output=True, text=True)
        assert r.returncode == 0  # every sum fits
        total = [a + float(b) for a, b in zip(total, r.stdout.split())]
    for d in range(3):
        assert total[2 * d + 1] <= total[2 * d], (d, total)
