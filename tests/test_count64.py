"""The grouped count that the mixed form takes again from the masses (counts past FP32), compiled for
the host from the kernels' own header: the FP64 form's floor(1e-4/psi), psi the rounded quotient, equal
for round ratios (1e-4/psi a whole number or an ulp beside it) and for any others."""
import subprocess

import numpy as np

from paper_2609_35967_gb300 import build

SRC = """
#include <cstdio>
#include "gd_ctx.h"
#include "gd_physics.cuh"
int main() {
  double a, b;
  while (std::scanf("%lf %lf", &a, &b) == 2) std::printf("%.17g\\n", gd::count64(a, b));
}
"""


def test_count_is_the_fp64_forms(tmp_path):
    src, exe = tmp_path / "count.cu", tmp_path / "count"
    src.write_text(SRC)
    subprocess.run([build._nvcc(), *build.FLAGS, "-I", build.CSRC, "-o", str(exe), str(src)], check=True)
    rng = np.random.default_rng(2)
    small = np.pi / 6 * 1.67 * rng.uniform(1e-4, 1e-3, 4000) ** 3
    ratio = np.concatenate([10.0 ** rng.integers(12, 18, 2000), 10.0 ** rng.uniform(12, 18, 2000)])
    big = small * ratio
    text = "".join(f"{a:.17g} {b:.17g}\n" for a, b in zip(big, small))
    run = subprocess.run([str(exe)], input=text, capture_output=True, text=True, check=True)
    got = np.array(run.stdout.split(), dtype=np.float64)
    assert np.array_equal(got, np.floor(1e-4 / (small / big)))
