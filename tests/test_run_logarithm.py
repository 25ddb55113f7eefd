"""The mixed form's |ln(m'/m)| of a run of events: compiled for the host from the kernels' own header.
The argument of log1p carries three FP32 roundings (difference, divisor, quotient) and its relative
error passes to the logarithm at most whole (x/((1 + x) ln(1 + x)) <= 1 for x >= 0); log1pf adds one
unit in the last place (2 u): 5 u, u = 2^-24, and 6 u with the second order, for losses as for growth."""
import subprocess

import numpy as np

from paper_2609_35967_gb300 import build

SRC = """
#include <cstdio>
#include "gd_ctx.h"
#include "gd_physics.cuh"
int main() {
  double a, b;
  while (std::scanf("%lf %lf", &a, &b) == 2) std::printf("%.9g\\n", (double)gd::abs_log_ratio(a, b));
}
"""


def test_run_logarithm_of_growth_and_loss(tmp_path):
    src, exe = tmp_path / "run_log.cu", tmp_path / "run_log"
    src.write_text(SRC)
    subprocess.run([build._nvcc(), *build.FLAGS, "-I", build.CSRC, "-o", str(exe), str(src)], check=True)
    rng = np.random.default_rng(1)
    m = 1e-12 * 10.0 ** rng.uniform(-2, 2, 600)
    F = np.concatenate([1.0 + 2.0 ** rng.uniform(-30, 0, 200), 10.0 ** rng.uniform(0, 9, 400)])
    for a, b in ((m, m * F), (m * F, m)):
        text = "".join(f"{u:.17g} {v:.17g}\n" for u, v in zip(a, b))
        run = subprocess.run([str(exe)], input=text, capture_output=True, text=True, check=True)
        got = np.array(run.stdout.split(), dtype=np.float64)
        ref = np.log1p(np.abs(b - a) / np.minimum(a, b))
        assert np.abs(got / ref - 1.0).max() < 6 * 2.0**-24
