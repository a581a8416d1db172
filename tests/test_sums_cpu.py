"""The device code's sums that also compile for the host, run on the CPU: errors against wider arithmetic."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2506_18408_gb300", "csrc")

# rms error of dot2 over that of one running sum (and of the sum in any of four interleaved chains), products of normal data
PROGRAM = r"""
#include "common.cuh"
#include <cmath>
#include <cstdio>
#include <random>
#include <vector>
int main() {
    std::mt19937_64 g(1);
    std::normal_distribution<double> nd;
    for (int n : {0, 1, 2, 3, 4, 5, 7, 8, 62, 63, 64, 100, 250, 1024}) {
        double e2 = 0, e1 = 0, worst = 0;
        for (int t = 0; t < 4000; ++t) {
            std::vector<double> x(3 * n + 3), y(n + 1);
            for (double& v : x) v = nd(g);
            for (double& v : y) v = nd(g);
            long double exact = 0, size = 0;
            double one = 0;
            for (int k = 0; k < n; ++k) {
                exact += (long double)x[3 * k] * y[k];
                size += std::fabs(x[3 * k] * y[k]);
                one = std::fma(x[3 * k], y[k], one);
            }
            const double got = sfg::dot2(x.data(), 3, y.data(), n);
            const double d2 = (double)(got - exact), d1 = (double)(one - exact);
            e2 += d2 * d2;
            e1 += d1 * d1;
            if (size > 0) worst = std::fmax(worst, std::fabs(d2) / (double)size);
        }
        std::printf("%d %.17g %.17g %.17g\n", n, std::sqrt(e2), std::sqrt(e1), worst);
    }
}
"""


def test_dot2_rounds_less_than_one_running_sum(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("no nvcc")
    src = tmp_path / "sums.cu"
    src.write_text(PROGRAM)
    exe = tmp_path / "sums"
    r = subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-std=c++17", "-O1", "-I", CSRC, "-o", str(exe),
                        str(src)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    for line in subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout.splitlines():
        n, e2, e1, worst = int(line.split()[0]), *map(float, line.split()[1:])
        # an entry passes at most ceil(n / 2) + 1 roundings, each of at most 2^-53 of the sizes added so far
        assert worst <= ((n + 1) // 2 + 1) * 2.0 ** -53 * 1.01
        # independent roundings: the error of a chain grows with its length's root (two chains: 0.71), after the join
        if n >= 62:
            assert e2 <= 0.85 * e1
