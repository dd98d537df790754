"""A small contraction step on its own (tests/small_step_check.cu): its sums, and that a zero factor hides
neither an infinity nor a NaN."""
import os
import subprocess

import pytest

from paper_2103_11595_gb300 import build_lib

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.mark.gpu
def test_small_step_sums_and_non_finite_factors(tmp_path):
    exe = str(tmp_path / "small_step_check")
    nvcc = os.path.join(build_lib.cuda_home(), "bin", "nvcc")
    subprocess.run([nvcc, build_lib.ARCH, "-O2", "-std=c++17", f"-I{build_lib.CSRC}",
                    os.path.join(HERE, "small_step_check.cu"), "-o", exe], check=True)
    out = subprocess.run([exe], check=True, capture_output=True, text=True).stdout
    rows = [tuple(map(int, line.split())) for line in out.splitlines()]
    assert rows == [(rk, 0, 0, 0) for rk in range(6)]  # none wrong, none of the row finite, none changed
