"""The FP32 near end of the K window against FP64: the bound on its error that
decides when the crack step takes its exact form (a column closer than that to
either end of the window) holds over the speeds and r0 that a lattice takes."""
import os
import subprocess

import paper_2206_12412_gb300 as pkg

SOURCE = r"""
#include "lbm_window.h"
#include <cmath>
#include <cstdio>
#include <random>
int main()
{
    std::mt19937_64 g(7);
    std::uniform_real_distribution<double> u(0.0, 1.0);
    double worst = 0.0;
    for (int k = 0; k < 20000000; ++k) {
        const double r0 = lbm::kWindowR0 * std::pow(20000.0, u(g));
        const double v_max = k % 3 == 0 ? u(g) : 1.0 - std::pow(10.0, -5.0 * u(g)), v = v_max * (k % 2 ? u(g) : 1.0 - 1e-3 * u(g));
        const float lo_max = (float)std::fmin((double)lbm::kWindowLo, 1.001 * r0 / (1.0 - v_max));
        const float lo_f = lbm::window_start((float)r0, v);
        if (!(lo_f < lo_max)) continue;   // the exact form is taken
        const long double lo = (long double)r0 / (1.0L - (long double)v) * 4294967296.0L;
        const long double err = fabsl((long double)(int64_t)(lo_f * 4294967296.0f) - lo);
        worst = fmax(worst, (double)(err / lbm::window_slack((float)r0, lo_max)));
    }
    std::printf("%.6f\n", worst);
}
"""


def test_window_start_error_bound(tmp_path):
    src, exe = tmp_path / "w.cc", tmp_path / "w"
    src.write_text(SOURCE)
    csrc = os.path.join(os.path.dirname(pkg.__file__), "csrc")
    subprocess.run(["g++", "-O2", "-std=c++17", "-I" + csrc, str(src), "-o", str(exe)], check=True)
    worst = float(subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout)
    assert 0.1 < worst < 1.0   # never beyond the bound, and the bound is no empty one
