"""The integer multiply-add under every FP64 product of the DG kernels (csrc/fx.cuh,
mad_wide): two instructions, of which the second still reads the factors, so the sum's
low word must not share a register with a factor of equal value."""
import os
import subprocess

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_factor_and_sum_of_equal_value(tmp_path):
    from paper_2510_00998_gb300 import build
    exe = str(tmp_path / "fx_mad")
    subprocess.run([build.nvcc(), "-std=c++17", "-O3", *build.ARCH, "-I" + build.CSRC,
                    os.path.join(ROOT, "tests", "fx_mad.cu"), "-o", exe], check=True)
    out = subprocess.run([exe], capture_output=True, text=True)
    assert out.returncode == 0 and out.stdout.split() == ["0"]
