"""Doubling by the exponent field (FP64 collision) against an addition, at both ends of the range and between."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
NVCC = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
PROGRAM = r"""
#include <cfloat>
#include <cmath>
#include <cstdio>
#include "lbe_block_sum.cuh"
int main() {
    const double v[] = {0.0, 4.9406564584124654e-324, 1.1e-310, DBL_MIN * 0.9999999, DBL_MIN, 1.0 / 3.0, 1.0, 2.5e7,
                        DBL_MAX / 4, DBL_MAX / 2, nextafter(DBL_MAX / 2, INFINITY), DBL_MAX, INFINITY};
    int bad = 0;
    for (double x : v)
        for (double s : {x, -x}) {
            const double t = lbe::twice(s), r = s + s;
            if (lbe::double_bits(t) != lbe::double_bits(r)) bad += std::printf("%g: %g, not %g\n", s, t, r) > 0;
        }
    if (!std::isnan(lbe::twice(NAN))) ++bad;
    return bad;
}
"""


@pytest.mark.skipif(not os.path.exists(NVCC), reason="needs nvcc (host code only)")
def test_twice(tmp_path):
    src = tmp_path / "twice.cu"
    src.write_text(PROGRAM)
    exe = str(tmp_path / "twice")
    subprocess.run([NVCC, "-std=c++20", "-O1", "--expt-relaxed-constexpr", "-gencode", "arch=compute_103a,code=sm_103a",
                    "-I", os.path.join(ROOT, "paper_1202_3842_gb300", "csrc"), str(src), "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
