"""The search for SpecTr's division factor (``spectr_root`` in analysis.cuh), compiled for the host."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
NVCC = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")

CODE = r"""
#include "analysis.cuh"
#include <cmath>
#include <cstdio>
#include <random>
#include <vector>
int main()
{
    std::mt19937 g(1);
    std::normal_distribution<double> nd;
    for (int k = 2; k <= 4; ++k)
        for (int rep = 0; rep < 60; ++rep) {
            const int V = rep % 2 ? 50 : 3000;
            std::vector<double> p(V), q(V);
            double sp = 0, sq = 0;
            for (int i = 0; i < V; ++i) {
                const double z = 2 * nd(g);
                q[i] = exp(z); p[i] = exp(z + nd(g));
                sp += p[i]; sq += q[i];
            }
            int n = 0;
            auto beta = [&](double r) { double b = 0; ++n; for (int i = 0; i < V; ++i) b += fmin(p[i] / sp / r, q[i] / sq); return b; };
            auto f = [&](double r) { const double b = beta(r); return 1 - pow(1 - b, k) - r * b; };
            const double x = specv::spectr_root((double)k, beta);
            const int evaluations = n;
            double lo = 1, hi = k;
            for (int i = 0; i < 60; ++i) { const double m = 0.5 * (lo + hi); (f(m) > 0 ? lo : hi) = m; }
            printf("%d %.17g %.17g %d\n", k, x, lo, evaluations);
        }
}
"""


@pytest.mark.skipif(shutil.which(NVCC) is None, reason="no nvcc")
def test_root_is_as_close_as_forty_halvings(tmp_path):
    """Within one final bracket, (k - 1) 2^-40, of 60 halvings (plus their own rounding, 1e-14), on laws for which the root is
    well conditioned; never more evaluations than two per halving and the two ends."""
    src, exe = tmp_path / "root.cu", tmp_path / "root"
    src.write_text(CODE)
    subprocess.check_call([NVCC, "-std=c++17", "-gencode", "arch=compute_100a,code=sm_100a", "-I", os.path.join(ROOT, "include"),
                           "-I", os.path.join(ROOT, "paper_2602_16994_b200", "csrc"), "-o", str(exe), str(src)], stderr=subprocess.DEVNULL)
    lines = subprocess.check_output([str(exe)], text=True).split("\n")[:-1]
    assert len(lines) == 180
    for line in lines:
        k, x, ref, n = line.split()
        assert abs(float(x) - float(ref)) <= (int(k) - 1) * 2.0**-40 + 1e-14, line
        assert int(n) <= 82, line
