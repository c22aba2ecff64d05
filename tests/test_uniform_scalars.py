"""The interval's and tolerances' scalars the host forms once per call: the
stage cap of a tolerance whose root is no int (undefined to convert) is the
largest int, on any host."""
import os
import subprocess

import pytest

from paper_1611_02274_gb300 import build as NB

SRC = r"""
#include <cstdio>
#include "common.cuh"
int main() {
    const double rtol[] = {1e-300, 1e-14, 1e-6, 1e-3, 1.0, 1e3, 1.02e4, 1.03e4, 1e6, 1e300};
    for (double r : rtol) printf("%d\n", bode::UniformScalars(0.0, 1.0, r, 0.0).mmax);
}
"""


def test_stage_cap_of_any_tolerance(tmp_path):
    src = tmp_path / "scalars.cu"
    src.write_text(SRC)
    exe = str(tmp_path / "scalars")
    try:
        cc = NB.nvcc()
    except RuntimeError:
        pytest.skip("needs nvcc")
    subprocess.run([cc, *NB.ARCH, "-std=c++17", "--expt-relaxed-constexpr", "-I", NB.INCLUDE, "-I", NB.CSRC, str(src), "-o", exe],
                   check=True, capture_output=True)
    out = [int(v) for v in subprocess.run([exe], check=True, capture_output=True, text=True).stdout.split()]
    u = 2.22e-16
    want = [max(2, round(min((r / (10 * u)) ** 0.5, 2.0 ** 31 - 1)))
            for r in (1e-300, 1e-14, 1e-6, 1e-3, 1.0, 1e3, 1.02e4, 1.03e4, 1e6, 1e300)]
    assert out == want
